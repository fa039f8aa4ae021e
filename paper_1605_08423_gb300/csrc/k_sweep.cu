// k_sweep.cu -- one Metropolis sweep of every walker (single-electron moves).
//
// For electron i (up block first, then down) with proposal r'_i (precomputed
// by the proposal kernel) and its orbital row phi'_j = phi_j(r'_i) (precomputed
// by the orbital kernel for the whole sweep):
//   ratio   R  = sum_j phi'_j G_{j,i}                     (determinant ratio)
//   Jastrow dU = sum_{j != i} [u_ee(r'_i,r_j) - u_ee(r_i,r_j)] + sum_a [u_en(r'_i,R_a) - u_en(r_i,R_a)]
//   accept if u < R^2 exp(2 dU)
// and on acceptance the Sherman-Morrison rank-1 update of the inverse of the
// spin block:  G' = G - G_{:,i} (phi'^T G - e_i^T) / R.
// The electron's own e-n sum V_i = sum_a u_en(r_i, R_a) is carried between the
// moves and the sweeps of a call (an accepted move replaces it by the sum at
// the proposal), so a move evaluates the e-n terms at the proposal only.
#include <algorithm>

#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// FP64 form, one warp per walker; the inverse of the moving spin block is
// staged in shared memory for the n moves of that block.
struct SweepSmem {
    // Rows of the staged inverse are 16-byte vectors: nv = n rounded up to a
    // whole vector (zero padded), row stride ld = nv + one vector, so that the
    // 16-byte accesses of 8 consecutive lanes (one per row) hit distinct banks.
    static constexpr int VE = 2;   // doubles per 16-byte vector
    __host__ __device__ static int nv(int n) { return (n + VE - 1) / VE * VE; }
    __host__ __device__ static int ld(int n) { return nv(n) + VE; }
    // per warp: G^T [n][ld], old row [nv], phi' [nv], proposal trig [6], trig
    // [6N], V [N], and only with the e-e-n-n Jastrow term (j34) three [N]
    // vectors (sum over electrons of chi_a, the same less the moving electron's,
    // and the change at its proposal); last the sums of two warps, [2][4]
    __host__ __device__ static size_t warp_bytes(int N, int n, bool j34) {
        size_t b = ((size_t)n * ld(n) + 2 * (size_t)nv(n) + 6) * sizeof(double);
        b += (size_t)(j34 ? 10 : 7) * N * sizeof(double) + 8 * sizeof(double);
        return (b + 15) & ~size_t(15);
    }
};

// exp(-zeta |d|^2) for the periodised displacement between two points given
// by their (sin, cos)(pi x / L) triples (e-e-n-n Jastrow orbital)
template <typename T>
__device__ __forceinline__ T jas_orbital(const T* a, const T* b, T ell, T zeta) {
    T t = 0;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const T sd = a[mu] * b[3 + mu] - a[3 + mu] * b[mu];
        t += sd * sd;
    }
    return qexp(-zeta * ell * ell * t);
}

template <typename T>
__device__ __forceinline__ T pair_dist(const T* a, const T* b, T ell) {
    // |d| for the periodised displacement between two points given by their
    // (sin, cos)(pi x / L) triples
    T t = 0;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const T sd = a[mu] * b[3 + mu] - a[3 + mu] * b[mu];
        t += sd * sd;
    }
    return ell * qsqrt_pair(t);
}

// Pade pair term c r / (1 + b r) of two points' trig triples (c = 1/2: e-e, c = -Zj: e-n).
__device__ __forceinline__ double pade_u(const double* a, const double* b, double ell, double cb, double cu) {
    const double r = pair_dist(a, b, ell);
    return cu * r * qrcp(fma(cb, r, 1.0));
}

// FP64 form.  Bound by the FP64 pipe (two multiply-adds a clock and SM, so a
// warp instruction occupies it for 16 clocks however many lanes are on): a move
// of N = 64 costs 3 N Pade pairs of 22 operations and the rank-1 update.  The
// new and old e-e terms share one lane loop of 2 N items, so that small N
// fills the warp; walkers are spread evenly over the SMs by the launcher.
// WW warps take a walker: one, or two where the walkers are so few that half of the
// SMs' four issue ports would idle (a port issues an FP64 instruction in 64 clocks,
// so a lone warp's move is a chain of some 90 of them at N = 16).  With two, the first
// takes the e-e terms, the second the ratio and the e-n terms, each summed in the order
// of the lone warp, and a row's update is cut over up to four threads: a walker's chain
// is the same to the bit whatever the number of walkers.  256 walkers of N = 16: 63 us a
// sweep, 80 with one warp.
template <int WW>
__global__ void __launch_bounds__(512) sweep_kernel(SysView<double> s, double* __restrict__ X,
                                                    const double* __restrict__ Xp, const double* __restrict__ ptp,
                                                    const double* __restrict__ uacc, const double* __restrict__ Phi,
                                                    double* __restrict__ Gt, unsigned long long* __restrict__ nacc,
                                                    double* __restrict__ Vep, int vep_init) {
    extern __shared__ __align__(16) unsigned char smraw[];
    constexpr int VE = SweepSmem::VE;
    const int N = s.N, n = s.n, nv = SweepSmem::nv(n), ld = SweepSmem::ld(n), nvv = nv / VE;
    constexpr int T = 32 * WW;
    const int lane = threadIdx.x & (T - 1), warp = threadIdx.x / T, wpb = blockDim.x / T;   // thread of the walker
    auto sync = [&]() {
        if (WW == 1) __syncwarp();
        else asm volatile("bar.sync %0, %1;\n" ::"r"(1 + warp), "n"(T) : "memory");
    };
    double* ptr_s = (double*)smraw;                          // [N][6] proton trig
    const size_t off = ((size_t)6 * N * sizeof(double) + 15) & ~size_t(15);
    const bool j34 = s.fjt != nullptr;
    unsigned char* mine = smraw + off + (size_t)warp * SweepSmem::warp_bytes(N, n, j34);
    double* Gs = (double*)mine;
    double* rowb = Gs + (size_t)n * ld;
    double* phi = rowb + nv;
    double* ptb = phi + nv;       // [6] the proposal's trig
    double* et = ptb + 6;
    double* vj = et + 6 * N;      // [N] V_i
    double* c34 = vj + N;         // [N] sum over electrons of chi_a (e-e-n-n Jastrow term)
    double* dif = c34 + N;        // [N] c_a - chi_a at the moving electron
    double* dch = dif + N;        // [N] change of chi_a at its proposal
    double* red = (double*)(mine + SweepSmem::warp_bytes(N, n, j34)) - 8;   // the warps' sums

    for (int idx = threadIdx.x; idx < 6 * N; idx += blockDim.x) ptr_s[idx] = s.ptrig[idx];
    __syncthreads();
    const int w = blockIdx.x * wpb + warp;
    if (w >= s.W) return;

    const double ell = s.ell, bee = s.b_ee, bep = s.b_ep, Zj = s.Zj;
    const double L = s.L, iL = s.iL;
    double* Xw = X + (size_t)w * 3 * N;   // positions stay in HBM; accepted moves are written through
    for (int idx = lane; idx < 3 * N; idx += T) {
        const int i = idx / 3, mu = idx % 3;
        double sn, cs;
        sincospi(Xw[idx] * iL, &sn, &cs);
        et[6 * i + mu] = sn;
        et[6 * i + 3 + mu] = cs;
    }
    sync();
    for (int i = lane; i < N; i += T) {
        double v = 0;
        if (vep_init)
            for (int a = 0; a < N; ++a) v += pade_u(et + 6 * i, ptr_s + 6 * a, ell, bep, -Zj);
        else
            v = Vep[(size_t)w * N + i];
        vj[i] = v;
    }
    const double zj = s.zeta_j;
    if (j34) {
        for (int a = lane; a < N; a += T) {
            double c = 0;
            for (int j = 0; j < N; ++j) c += jas_orbital(et + 6 * j, ptr_s + 6 * a, ell, zj);
            c34[a] = c;
        }
    }
    sync();
    for (int j = n + lane; j < nv; j += T) phi[j] = 0.0;   // padding stays zero
    unsigned long long naccept = 0;
    // the next move's proposal trig (lanes 0-5), orbital row (n <= 64: two per
    // lane) and uniform are loaded one move ahead, so their HBM latency
    // overlaps a move
    double pt_nx, ph_nx[2], u_nx;
    auto fetch = [&](int i) {
        const size_t row = (size_t)w * N + i;
        pt_nx = lane < 6 ? ptp[row * 6 + lane] : 0.0;
#pragma unroll
        for (int k = 0; k < 2; ++k) ph_nx[k] = (lane + T * k < n) ? Phi[row * n + lane + T * k] : 0.0;
        u_nx = uacc[row];
    };
    fetch(0);
    for (int sp = 0; sp < 2; ++sp) {
        double* G = Gt + ((size_t)w * 2 + sp) * n * n;
        for (int idx = lane; idx < n * nv; idx += T) {
            const int r = idx / nv, c = idx - r * nv;
            Gs[r * ld + c] = c < n ? G[r * n + c] : 0.0;
        }
        sync();
        for (int il = 0; il < n; ++il) {
            const int i = sp * n + il;
            const size_t row = (size_t)w * N + i;
            if (lane < 6) ptb[lane] = pt_nx;
#pragma unroll
            for (int k = 0; k < 2; ++k)
                if (lane + T * k < n) phi[lane + T * k] = ph_nx[k];
            const double u = u_nx;
            if (i + 1 < N) fetch(i + 1);
            sync();
            // items 0..N-1: u_ee at the proposal, N..2N-1: minus u_ee at the old position
            const double* ei = et + 6 * i;
            const int ln = lane & 31;
            double part = 0, du = 0, vnew = 0;
            if (WW == 1 || lane < 32)
                for (int k = ln; k < 2 * N; k += 32) {
                    const bool old = k >= N;
                    const int j = old ? k - N : k;
                    const double v = pade_u(old ? ei : ptb, et + 6 * j, ell, bee, old ? -0.5 : 0.5);
                    du += j != i ? v : 0.0;
                }
            if (WW == 1 || lane >= 32) {
                for (int j = ln; j < n; j += 32) part += phi[j] * Gs[il * ld + j];
                for (int a = ln; a < N; a += 32) vnew += pade_u(ptb, ptr_s + 6 * a, ell, bep, -Zj);
            }
            if (j34) {
                // e-e-n-n term: the pairs (i, j != i) change by
                // sum_a (chi_a(r'_i) - chi_a(r_i)) sum_b f_ab (c_b - chi_b(r_i))
                for (int a = lane; a < N; a += T) {
                    const double old = jas_orbital(ei, ptr_s + 6 * a, ell, zj);
                    dch[a] = jas_orbital(ptb, ptr_s + 6 * a, ell, zj) - old;
                    dif[a] = c34[a] - old;
                }
                sync();
                for (int a = lane; a < N; a += T) {
                    // f is symmetric (checked at qmc_init): column a = row a,
                    // and the lanes' loads of a column element are consecutive
                    const double* fa = s.fjt + a;
                    double wa = 0;
                    for (int b = 0; b < N; ++b) wa += fa[(size_t)b * N] * dif[b];
                    du += dch[a] * wa;
                }
            }
            // the three warp sums in seven additions: the halves of the warp exchange
            // (ratio, du) for (vnew, 0), then the quarters
            double ratio;
            if (WW == 1) {
                const bool hi = lane & 16, qr = lane & 8;
                double a0 = hi ? vnew : part, a1 = hi ? 0.0 : du;
                a0 += __shfl_xor_sync(0xffffffffu, hi ? part : vnew, 16);
                a1 += __shfl_xor_sync(0xffffffffu, hi ? du : 0.0, 16);
                double x = qr ? a1 : a0;
                x += __shfl_xor_sync(0xffffffffu, qr ? a0 : a1, 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                ratio = __shfl_sync(0xffffffffu, x, 0);
                du = __shfl_sync(0xffffffffu, x, 8);
                vnew = __shfl_sync(0xffffffffu, x, 16);
            } else {         // du is the first warp's, ratio and vnew the second's; each added up in the same order
                const bool hi = lane & 16, second = lane >= 32;
                double x = second ? (hi ? vnew : part) : du;
                x += __shfl_xor_sync(0xffffffffu, second ? (hi ? part : vnew) : du, 16);
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
                double* rd = red + 4 * (il & 1);     // alternating: read after the barrier, written a move later
                if ((lane & 15) == 0) rd[lane >> 4] = x;
                sync();
                du = rd[0];
                ratio = rd[2];
                vnew = rd[3];
            }
            du += vnew - vj[i];
            const double prob = ratio * ratio * qexp(2.0 * du);
            if (u < prob) {
                for (int j = lane; j < nv; j += T) rowb[j] = Gs[il * ld + j];
                sync();
                const double ir = qrcp(ratio);
                const double2* phv = (const double2*)phi;
                const double2* rbv = (const double2*)rowb;
                // two warps: S consecutive threads per row, which update every S-th vector each
                const int S = WW == 1 ? 1 : n <= 16 ? 4 : n <= 32 ? 2 : 1, h = lane & (S - 1);
                for (int l = lane / S; l < n; l += T / S) {
                    double2* gl = (double2*)(Gs + l * ld);
                    double w0 = 0, w1 = 0;   // two partial sums: short chains
                    for (int jv = 0; jv < nvv; ++jv) {
                        const double2 p = phv[jv], g = gl[jv];
                        w0 += p.x * g.x; w1 += p.y * g.y;
                    }
                    const double coef = ((w0 + w1) - (l == il ? 1.0 : 0.0)) * ir;
                    if (S > 1) __syncwarp(((1u << S) - 1u) << (lane & 31 & ~(S - 1)));   // the row's threads have read it
                    for (int jv = h; jv < nvv; jv += S) {
                        const double2 g = gl[jv], r = rbv[jv];
                        gl[jv] = make_double2(g.x - coef * r.x, g.y - coef * r.y);
                    }
                }
                if (lane < 3) {   // wrap into [0, L) at once (as the reference chain does)
                    const double xpl = Xp[row * 3 + lane];
                    const double q = xpl * iL, f = floor(q);
                    // the division only where the product's rounding could decide
                    Xw[3 * i + lane] = xpl - L * (fabs(q - rint(q)) > 1e-12 ? f : floor(xpl / L));
                }
                // the trig triple of the unwrapped proposal: wrapping flips the
                // signs of a component's sine and cosine together, and every use
                // is even in that sign
                if (lane < 6) et[6 * i + lane] = ptb[lane];
                if (lane == 0) vj[i] = vnew;
                if (j34)
                    for (int a = lane; a < N; a += T) c34[a] += dch[a];
                ++naccept;
            }
            sync();
        }
        for (int idx = lane; idx < n * n; idx += T) G[idx] = Gs[(idx / n) * ld + idx % n];
        sync();
    }
    for (int i = lane; i < N; i += T) Vep[(size_t)w * N + i] = vj[i];
    if (lane == 0) nacc[w] += naccept;
}


// Mixed form, n <= 64: two warps per walker and the inverse in registers.
// Thread tw (0..63) of a walker owns row tw of the staged inverse (G^T row,
// zero-padded to 64 columns), so a move touches no shared-memory copy of G:
//   w_l = sum_j phi'_j G^T[l][j] for every row (the ratio is w_il),
//   on acceptance every thread applies G^T[l] -= (w_l - delta_{l,il}) / R * G^T[il].
// The Jastrow difference is split over the 64 threads (two e-e and two e-n
// partners each).  The two warps of a walker meet at a named barrier (one
// per walker of the CTA), once per move: before it every thread has put its
// share of the Jastrow difference, the owner of row il its row and w_il, and
// every thread its element of the next move's orbital row into shared
// buffers that alternate between moves; after it the acceptance decision and
// the update need nothing else.  Electron i's (sin, cos) after an accepted
// move are written by the thread that has i among its partners (tw = i mod
// 64), the only thread that reads them later in the sweep.  Same proposals, uniforms and acceptance rule as
// sweep_kernel; the mixed form keeps accepted proposals unwrapped.
// With the e-e-n-n Jastrow term (s.fjt set) the CTA stages f (FP32, N x N) in
// shared memory and each walker keeps c_a = sum_j chi_a(r_j); a move of
// electron i changes U by sum_a (chi_a(r'_i) - chi_a(r_i)) w_a with
// w_a = sum_b f_ab (c_b - chi_b(r_i)), each thread taking nuclei tw and
// tw + 64 (one more barrier per move to publish c_b - chi_b(r_i), which the owner of
// b forms once: 270 -> 240 us a sweep of 1501 walkers, N = 54).
constexpr int kSwWalkers = 4;   // walkers per CTA (8 warps)
constexpr int kSwRow = 64;      // register row length (n <= 64)

// Stride of one point's (sin, cos)(pi x / L) triples in sweep_reg_kernel's
// shared memory: 7 floats, so that the 32 lanes reading 32 consecutive points
// hit 32 distinct banks (a stride of 6 pairs them up).
constexpr int kTS = 7;

// Shared-memory floats per walker of sweep_reg_kernel: phi [2][64], row
// [2][64], red [2][8], trig [kTS N], V [N], and with the e-e-n-n term c [N]
// and c - chi(r_i) [N]; rounded up to whole 16-byte vectors (phi and the row are
// read as float4).
__host__ __device__ inline size_t sweep_reg_walker_floats(int N, bool j34) {
    return (4 * kSwRow + 16 + (kTS + 1) * (size_t)N + (j34 ? 2 * (size_t)N + 3 : 0) + 3) & ~size_t(3);
}

__global__ void __launch_bounds__(64 * kSwWalkers) sweep_reg_kernel(SysView<float> s, double* __restrict__ X,
                                                                  const double* __restrict__ Xp,
                                                                  const float* __restrict__ ptp,
                                                                  const float* __restrict__ uacc,
                                                                  const float* __restrict__ Phi,
                                                                  float* __restrict__ Gt,
                                                                  unsigned long long* __restrict__ nacc,
                                                                  float* __restrict__ Vep, int vep_init) {
    extern __shared__ __align__(16) unsigned char smraw[];
    const int N = s.N, n = s.n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int p = warp >> 1, h = warp & 1, tw = tid & 63;
    const bool j34 = s.fjt != nullptr;
    float* ptr_s = (float*)smraw;                                       // [N][kTS] proton trig
    float* f_s = ptr_s + ((kTS * N + 3) & ~3);                            // [N][N] e-e-n-n coefficients (j34)
    float* mine = f_s + (j34 ? (size_t)N * N : 0) + (size_t)p * sweep_reg_walker_floats(N, j34);
    float* phi = mine;                  // [2][64] orbital row at the proposal (zero beyond n)
    float* rowb = phi + 2 * kSwRow;     // [2][64] row il of G^T
    float* red = rowb + 2 * kSwRow;     // [2][8] e-e du halves, ratio, new e-n sum halves
    float* dif = red + 16;              // [N] c_a - chi_a at the moving electron (j34; 16-byte aligned)
    float* et = dif + (j34 ? (N + 3) & ~3 : 0);   // [N][kTS] (sin, cos)(pi x / L) of the current positions
    float* vj = et + kTS * N;           // [N] V_i = sum_a u_en(r_i, R_a) at the current positions
    float* c34 = vj + N;                // [N] sum_j chi_a(r_j) (j34)
    for (int idx = tid; idx < 6 * N; idx += blockDim.x) ptr_s[kTS * (idx / 6) + idx % 6] = s.ptrig[idx];
    if (j34)
        for (int idx = tid; idx < N * N; idx += blockDim.x) f_s[idx] = s.fjt[idx];
    __syncthreads();
    const int w = blockIdx.x * kSwWalkers + p;
    if (w >= s.W) return;              // whole walkers only: both of its warps leave
    auto bar = [&]() { asm volatile("bar.sync %0, 64;\n" ::"r"(1 + p) : "memory"); };

    const float ell = (float)s.ell, bee = (float)s.b_ee, bep = (float)s.b_ep, Zj = (float)s.Zj;
    const double iL = 1.0 / s.L;
    double* Xw = X + (size_t)w * 3 * N;
    for (int idx = tw; idx < 3 * N; idx += 64) {
        const int i = idx / 3, mu = idx % 3;
        float sn, cs;
        sincospif((float)(Xw[idx] * iL), &sn, &cs);
        et[kTS * i + mu] = sn;
        et[kTS * i + 3 + mu] = cs;
    }
    const float zj = (float)s.zeta_j;
    bar();   // et complete
    // V_i: computed from the positions in the first sweep of a call, carried
    // in Vep between the call's sweeps (an accepted move sets V_i to the sum
    // of its new e-n terms), so a move evaluates the e-n Pade terms only at
    // the proposal
    for (int i = tw; i < N; i += 64) {
        float v = 0.f;
        if (vep_init) {
            for (int a = 0; a < N; ++a) {
                float u0, d1, d2, d3;
                pade_ep(bep, Zj, pair_dist(et + kTS * i, ptr_s + kTS * a, ell), u0, d1, d2, d3);
                v += u0;
            }
        } else {
            v = Vep[(size_t)w * N + i];
        }
        vj[i] = v;
    }
    if (j34) {
        for (int a = tw; a < N; a += 64) {
            float c = 0.f;
            for (int j = 0; j < N; ++j) c += jas_orbital(et + kTS * j, ptr_s + kTS * a, ell, zj);
            c34[a] = c;
        }
    }
    // proposal trig and uniform of a row; the orbital value phi_tw of a row
    auto ld_pt = [&](int i, float* pt_, float& u_) {
        const size_t row = (size_t)w * N + i;
#pragma unroll
        for (int mu = 0; mu < 6; ++mu) pt_[mu] = ptp[row * 6 + mu];
        u_ = uacc[row];
    };
    auto ld_ph = [&](int i) { return tw < n ? Phi[((size_t)w * N + i) * n + tw] : 0.f; };
    unsigned long long naccept = 0;
    const bool vec4 = (n & 3) == 0;
    for (int sp = 0; sp < 2; ++sp) {
        float* G = Gt + ((size_t)w * 2 + sp) * n * n;
        float g[kSwRow];
#pragma unroll
        for (int jv = 0; jv < kSwRow / 4; ++jv) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            const int j = 4 * jv;
            if (tw < n && j < n) {
                if (vec4) {
                    v = *(const float4*)(G + (size_t)tw * n + j);
                } else {
                    v.x = G[(size_t)tw * n + j];
                    if (j + 1 < n) v.y = G[(size_t)tw * n + j + 1];
                    if (j + 2 < n) v.z = G[(size_t)tw * n + j + 2];
                    if (j + 3 < n) v.w = G[(size_t)tw * n + j + 3];
                }
            }
            g[j] = v.x; g[j + 1] = v.y; g[j + 2] = v.z; g[j + 3] = v.w;
        }
        const int i0 = sp * n;
        phi[tw] = ld_ph(i0);                      // the spin's first move: buffer 0
        float ph_nx = n > 1 ? ld_ph(i0 + 1) : 0.f;   // the next move's value, stored during this move
        float pt_nx[6], u_nx;
        ld_pt(i0, pt_nx, u_nx);
        bar();   // buffer 0 and the positions visible; the previous spin's reads done
        for (int il = 0; il < n; ++il) {
            const int i = i0 + il, buf = il & 1;
            const size_t row = (size_t)w * N + i;
            float pt[6];
#pragma unroll
            for (int mu = 0; mu < 6; ++mu) pt[mu] = pt_nx[mu];
            const float u = u_nx;
            const float ph_wr = ph_nx;
            if (il + 1 < n) ld_pt(i + 1, pt_nx, u_nx);
            if (il + 2 < n) ph_nx = ld_ph(i + 2);
            // w_l for this thread's row: four partial sums
            const float4* phv = (const float4*)(phi + buf * kSwRow);
            float a4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int jv = 0; jv < kSwRow / 4; ++jv) {
                const float4 ph = phv[jv];
                a4[0] += ph.x * g[4 * jv]; a4[1] += ph.y * g[4 * jv + 1];
                a4[2] += ph.z * g[4 * jv + 2]; a4[3] += ph.w * g[4 * jv + 3];
            }
            const float wl = (a4[0] + a4[1]) + (a4[2] + a4[3]);
            // Jastrow difference: partners tw and tw + 64 (e-e: new minus old
            // pair terms; e-n: the new terms, less V_i after the barrier)
            float du = 0.f, vnew = 0.f;
            const float* ei = et + kTS * i;
#pragma unroll
            for (int k = 0; k < 2; ++k) {
                const int j = tw + 64 * k;
                if (j < N) {
                    const float* ej = et + kTS * j;
                    float u1, u0, d1, d2;
                    pade_ee(bee, pair_dist(pt, ej, ell), u1, d1, d2);
                    pade_ee(bee, pair_dist(ei, ej, ell), u0, d1, d2);
                    du += (j != i) ? u1 - u0 : 0.f;
                    const float* pa = ptr_s + kTS * j;
                    float d3;
                    pade_ep(bep, Zj, pair_dist(pt, pa, ell), u1, d1, d2, d3);
                    vnew += u1;
                }
            }
            float chn_r[2] = {0.f, 0.f}, cho_r[2] = {0.f, 0.f};
            if (j34) {
                // chi_a at the electron and at its proposal for this thread's nuclei
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int a = tw + 64 * k;
                    if (a < N) {
                        chn_r[k] = jas_orbital(pt, ptr_s + kTS * a, ell, zj);
                        cho_r[k] = jas_orbital(ei, ptr_s + kTS * a, ell, zj);
                        dif[a] = c34[a] - cho_r[k];
                    }
                }
                bar();   // c_b - chi_b(r_i) of every nucleus visible
#pragma unroll
                for (int k = 0; k < 2; ++k) {
                    const int a = tw + 64 * k;
                    if (a < N) {
                        float wa = 0.f;
                        int b = 0;
                        for (; b + 4 <= N; b += 4) {
                            const float4 d = *(const float4*)(dif + b);
                            wa += f_s[(size_t)b * N + a] * d.x;
                            wa += f_s[(size_t)(b + 1) * N + a] * d.y;
                            wa += f_s[(size_t)(b + 2) * N + a] * d.z;
                            wa += f_s[(size_t)(b + 3) * N + a] * d.w;
                        }
                        for (; b < N; ++b) wa += f_s[(size_t)b * N + a] * dif[b];
                        du += (chn_r[k] - cho_r[k]) * wa;
                    }
                }
            }
            du = warp_sum(du);
            vnew = warp_sum(vnew);
            float* rd = red + 8 * buf;
            float* rb = rowb + buf * kSwRow;
            if (lane == 0) { rd[h] = du; rd[4 + h] = vnew; }
            if (tw == il) {
                rd[2] = wl;
#pragma unroll
                for (int jv = 0; jv < kSwRow / 4; ++jv)
                    ((float4*)rb)[jv] = make_float4(g[4 * jv], g[4 * jv + 1], g[4 * jv + 2], g[4 * jv + 3]);
            }
            if (il + 1 < n) phi[(buf ^ 1) * kSwRow + tw] = ph_wr;
            const float v_old = vj[i];   // before the barrier: an accepted move rewrites it after
            bar();
            const float ratio = rd[2];
            const float vin = rd[4] + rd[5];
            const float dut = (rd[0] + rd[1]) + (vin - v_old);
            const float prob = ratio * ratio * expf(2.f * dut);
            if (u < prob) {
                const float coef = (wl - (tw == il ? 1.f : 0.f)) * __fdividef(1.f, ratio);
                const float4* rbv = (const float4*)rb;
#pragma unroll
                for (int jv = 0; jv < kSwRow / 4; ++jv) {
                    const float4 r4 = rbv[jv];
                    g[4 * jv] -= coef * r4.x; g[4 * jv + 1] -= coef * r4.y;
                    g[4 * jv + 2] -= coef * r4.z; g[4 * jv + 3] -= coef * r4.w;
                }
                // keep the proposal as is (periodic functions; the next proposal pass wraps)
                if (tw < 3) Xw[3 * i + tw] = Xp[row * 3 + tw];
                if (tw == (i & 63)) {
#pragma unroll
                    for (int mu = 0; mu < 6; ++mu) et[kTS * i + mu] = pt[mu];
                    vj[i] = vin;   // read again only in the next sweep
                }
                if (j34) {      // c_a of this thread's nuclei (read by others only after the next barrier)
#pragma unroll
                    for (int k = 0; k < 2; ++k) {
                        const int a = tw + 64 * k;
                        if (a < N) c34[a] += chn_r[k] - cho_r[k];
                    }
                }
                ++naccept;
            }
        }
        if (tw < n) {
#pragma unroll
            for (int j = 0; j < kSwRow; ++j)
                if (j < n) G[(size_t)tw * n + j] = g[j];
        }
    }
    bar();   // the last accepted moves' V_i
    for (int i = tw; i < N; i += 64) Vep[(size_t)w * N + i] = vj[i];
    if (tw == 0) nacc[w] += naccept;
}

static int sm_count() {
    static const int sms = [] {
        int dev = 0, v = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
        return v > 0 ? v : 1;
    }();
    return sms;
}

// Walkers per CTA of a kernel that takes one warp per walker: at most `most`
// (shared memory), and no more than spreads the walkers evenly over the SMs in
// the fewest rounds.  With 16 walkers a CTA, 1024 walkers sat on 64 of the 152
// SMs and a sweep of N = 64 took 2.9 ms (0.9 ms with 7 a CTA on 147 of them).
int walkers_per_cta(int W, int most) {
    const int sms = sm_count();
    const long long per_round = (long long)sms * most;
    const long long rounds = (W + per_round - 1) / per_round;
    return (int)((W + sms * rounds - 1) / (sms * rounds));
}

void launch_sweep(const SysView<float>& s, double* X, const double* Xp, const float* ptp, const float* uacc,
                  const float* Phi, float* Gt, unsigned long long* nacc, float* vep, bool vep_init, cudaStream_t st) {
    const bool j34 = s.fjt != nullptr;
    const size_t smem = sizeof(float) * (((kTS * s.N + 3) & ~3) + (j34 ? (size_t)s.N * s.N : 0) +
                                         kSwWalkers * sweep_reg_walker_floats(s.N, j34));
    static size_t attr = 0;
    if (smem > attr &&
        cudaFuncSetAttribute(sweep_reg_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess)
        attr = smem;
    sweep_reg_kernel<<<(s.W + kSwWalkers - 1) / kSwWalkers, 64 * kSwWalkers, smem, st>>>(s, X, Xp, ptp, uacc, Phi, Gt,
                                                                                         nacc, vep, vep_init ? 1 : 0);
}

void launch_sweep(const SysView<double>& s, double* X, const double* Xp, const double* ptp, const double* uacc,
                  const double* Phi, double* Gt, unsigned long long* nacc, double* vep, bool vep_init,
                  cudaStream_t st) {
    const size_t wb = SweepSmem::warp_bytes(s.N, s.n, s.fjt != nullptr);
    const size_t head = ((size_t)6 * s.N * sizeof(double) + 15) & ~size_t(15);
    const int fit = (int)((226 * 1024 - head) / wb);
    const int wpb = walkers_per_cta(s.W, std::max(1, std::min(16, fit)));
    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(sweep_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        cudaFuncSetAttribute(sweep_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        attr_set = true;
    }
    // two warps a walker while they still find a free issue port each: at most two walkers
    // an SM, and no other trajectory's kernels beside them (six served trajectories of
    // 256 walkers: 10.6 ms a step, 10.4 with one warp); the e-e-n-n sums stay with one warp
    if (wpb <= 2 && s.W <= 2 * sm_count() && !s.served && !s.fj)
        sweep_kernel<2><<<(s.W + wpb - 1) / wpb, 64 * wpb, head + wpb * wb, st>>>(s, X, Xp, ptp, uacc, Phi, Gt, nacc, vep,
                                                                                  vep_init ? 1 : 0);
    else
        sweep_kernel<1><<<(s.W + wpb - 1) / wpb, 32 * wpb, head + wpb * wb, st>>>(s, X, Xp, ptp, uacc, Phi, Gt, nacc, vep,
                                                                                  vep_init ? 1 : 0);
}

}  // namespace qmc
