// k_measure64.cu -- local energy and nuclear-force sample of every walker, FP64
// form (the mixed form's kernel and the estimators are in k_measure.cu).
//
// One CTA per walker.  The FP64 pipe bounds everything here (an SM issues a warp's
// FP64 instruction every 16 clocks), so the kernel is arranged for few FP64
// operations.  The orbital rows D = grad phi and Lp = lap phi are not needed:
// with C the coefficients, G the inverse of a spin block and Z = C G,
//   g_i = sum_b Z_bi grad chi_b(r_i),   l_i = sum_b Z_bi lap chi_b(r_i),
//   y_bi = -1/2 lap chi_b(r_i) - grad_i U . grad chi_b(r_i),
//   M = y^T Z (= Y G with Y_ij = sum_b y_bi C_bj),   P = Z M (= C G Y G),
// three B x n x n products per spin and one pass over the basis, where forming
// D, Lp (five products) and then Z, K = G Y G and P took seven and two n^3 ones,
// two passes over the basis and 4 N n doubles a walker through memory.  The
// radial chain of a Gaussian enters through s_q = sum_g Z_bi (-zeta_g)^q chi_b, so
// a Gaussian costs its exponential and about ten operations, and the geometry is
// done once per (nucleus, electron):
//   grad: 2 s1 p;   lap: 4 s2 |p|^2 + 2 s1 sum q;
//   H gU + 1/2 grad lap:  p (4 s2 p.gU + 4 s3 |p|^2 + 2 s2 sum q - k2 s1 + 4 s2 q) + 2 s1 q o gU.
// N = 64, 1024 walkers: orbital rows + sample 12.1 ms before, 6.8 ms now (7.2 with the
// e-e Jastrow pairs evaluated from both ends).
//
// Twisted form (complex Bloch-summed orbitals, k_twist.cu): the same with complex
// G, y and real C, so there Y_ij = sum_b y_bi C_bj, K = G Y G and P = C K are the
// cheaper products (6 B n^2 + 8 n^3 real multiply-adds a spin, 10 B n^2 through M).
// The orbitals factorise over the axes, chi = e^{i theta.k} s_x s_y s_z, and with
// D = grad_i U . grad + 1/2 lap = D_x + D_y + D_z,
//   y = -D chi,   H gU + 1/2 grad lap = grad (D chi),
// everything follows from s_q = d^q s, t = D_mu s and t' = d D_mu s of each axis.
// N = 64, 512 walkers: rows + g, l + sample + force terms 15.5 ms before in four
// kernels, 9.2 ms now in one.
#include "bloch.cuh"
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

namespace {

constexpr int kThreads = 256, kWarps = kThreads / 32;

int pad_pow2(int n) {
    int p = 4;
    while (p < n) p *= 2;
    return p;
}

// Shared memory of one CTA.  tb: basis rows per tile; in the real form with tb >= B
// the Z and chi rows of a spin block stay for the second pass.  The twisted form
// keeps G in shared memory up to n = 32 (np <= 32) and reads it from global memory above.
// rho(k) stands behind the phase table in the work space of the orbital products, which
// are done by then: at the largest cutoff (ewald_mmax = 12, 3576 vectors) its 57 KB beside
// them left no launch for twisted cells of N >= 84 (every accepted cell fits 225 KB now).
struct M64Layout {
    size_t xs, et, gU, lU, Ui, gi, vv, li, facc, rhot, red, part, uni, total;
    __host__ __device__ static size_t square2(int np) { return (size_t)np * (2 * np + 4); }   // complex np x np, planar
    __host__ __device__ M64Layout(int N, int n, int np, int nk, int mmax, bool tw, bool j34, int tb) {
        size_t o = 0;
        auto take = [&](size_t doubles) { const size_t r = o; o = (o + 8 * doubles + 15) & ~size_t(15); return r; };
        xs = take(3 * N); et = take(6 * N); gU = take(3 * N); lU = take(N); Ui = take(N);
        gi = take(3 * N); vv = take(3 * N); li = take(N);
        facc = take(9 * N);
        red = take(64);
        // slices of the Jastrow sums (5 + 4 per electron; N <= kThreads), then the warps' g_i, l_i sums
        const size_t jp = 9 * (size_t)kThreads, gp = 4 * (size_t)kWarps * n;
        part = take(jp > gp ? jp : gp);
        const size_t table = 2 * (size_t)N * 3 * (mmax + 1);                  // phase table
        size_t u = table + 2 * (size_t)nk;
        if (tw) {
            const size_t sq = square2(np), tile = (size_t)tb * (2 * np + 2);
            const size_t s = (np <= 32 ? 2 : 1) * sq + (sq > tile ? sq : tile);       // G, Y / K, then T or the tile
            u = u > s ? u : s;
        } else {
            const size_t s = 2 * (size_t)np * (np + 2) + 3 * (size_t)tb * (np + 2);   // G, M, Z, chi, y / P
            u = u > s ? u : s;
        }
        if (j34 && 92 * (size_t)N > u) u = 92 * (size_t)N;   // c, S, 5 a warp, the warps' force terms
        uni = take(u);
        rhot = uni + 8 * table;
        total = o;
    }
};

// Basis rows per tile: the whole spin block if it fits (one tile, nothing evaluated
// twice), else as many whole nuclei as do, but full rounds of 4 x 4 outputs over the
// threads (64 rows at n > 32, 128 at n <= 32; half of that in the twisted form).
// N = 128, four Gaussians, 608 walkers: 29.5 ms so, 36.0 with the 68 rows that fit (272
// tasks: a second round for 16 of them); one to three Gaussians 15.3, 20.0 and 25.2 where
// all rows that fit take 16.2, 22.4 and 28.7.
int tile_rows(int N, int n, int G, int nk, int mmax, bool tw, bool j34) {
    const int np = pad_pow2(n);
    const size_t most = 225 * 1024;
    int rows = N * G;
    while (rows > G && M64Layout(N, n, np, nk, mmax, tw, j34, rows).total > most) rows -= G;
    const int round = 16 * kThreads / (tw ? 2 * np : np);
    if (rows < N * G && rows > round) rows = rows / round * round / G * G;
    return rows;
}

// Periodised geometry of electron trig e and nucleus trig a: p, q, t (sin, cos
// of the difference from the two points' values; q = cos^2 - sin^2 = 1 - 2 sin^2).
struct Geo { double p[3], q[3], t; };
__device__ __forceinline__ Geo geometry(const double* e, const double* a, double ell) {
    Geo g;
    double s2 = 0;
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        const double sd = e[mu] * a[3 + mu] - e[3 + mu] * a[mu];
        const double cd = e[3 + mu] * a[3 + mu] + e[mu] * a[mu];
        const double ss = sd * sd;
        g.p[mu] = ell * sd * cd;
        g.q[mu] = fma(-2.0, ss, 1.0);
        s2 += ss;
    }
    g.t = ell * ell * s2;
    return g;
}

// Sums of nv values within segments of seg < 32 lanes (a power of two).
__device__ __forceinline__ void seg_sum(double* v, int nv, int seg) {
    for (int k = 0; k < nv; ++k)
        for (int o = seg >> 1; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
}

// out[r][i] (r < rows) = sum_{j < kk} A(r, j) Bm[j][i], TT x TT outputs a thread.
// A rows from global memory with row stride lda (Z = C G) or shared (P = Z M).
template <int TT>
__device__ __forceinline__ void product(int rows, int np, int kk, const double* __restrict__ A, int lda, int rmax,
                                        const double* Bm, int ldb, double* out, int ldo) {
    const int ncg = np / TT, tasks = (rows + TT - 1) / TT * ncg;
    for (int task = threadIdx.x; task < tasks; task += kThreads) {
        const int r0 = task / ncg * TT, c0 = task % ncg * TT;
        const double* ar[TT];
#pragma unroll
        for (int a = 0; a < TT; ++a) ar[a] = A + (size_t)(r0 + a < rmax ? r0 + a : rmax - 1) * lda;
        double acc[TT][TT] = {};
#pragma unroll 2
        for (int j = 0; j < kk; ++j) {
            double bv[TT];
#pragma unroll
            for (int b = 0; b < TT; ++b) bv[b] = Bm[j * ldb + c0 + b];
#pragma unroll
            for (int a = 0; a < TT; ++a) {
                const double av = ar[a][j];
#pragma unroll
                for (int b = 0; b < TT; ++b) acc[a][b] += av * bv[b];
            }
        }
#pragma unroll
        for (int a = 0; a < TT; ++a)
            if (r0 + a < rows)
#pragma unroll
                for (int b = 0; b < TT; ++b) out[(r0 + a) * ldo + c0 + b] = acc[a][b];
    }
}
__device__ __forceinline__ void product_any(int rows, int np, int kk, const double* A, int lda, int rmax,
                                            const double* Bm, int ldb, double* out, int ldo) {
    // 4 x 4 outputs a thread where that fills the CTA (fewest shared-memory reads), else 2 x 2
    if ((rows / 4) * (np / 4) >= kThreads / 2) product<4>(rows, np, kk, A, lda, rmax, Bm, ldb, out, ldo);
    else product<2>(rows, np, kk, A, lda, rmax, Bm, ldb, out, ldo);
}

// M[i'][i] += sum_{b < rows} y[b][i'] Z[b][i], TT x TT of the np x np outputs a thread, kept in acc.
template <int TT>
__device__ __forceinline__ void gram_acc(int rows, int np, const double* y, const double* Z, int ld, double* acc) {
    const int ng = np / TT;
    if ((int)threadIdx.x >= ng * ng) return;
    const int r0 = threadIdx.x / ng * TT, c0 = threadIdx.x % ng * TT;
#pragma unroll 2
    for (int b = 0; b < rows; ++b) {
        double yv[TT], zv[TT];
#pragma unroll
        for (int a = 0; a < TT; ++a) { yv[a] = y[b * ld + r0 + a]; zv[a] = Z[b * ld + c0 + a]; }
#pragma unroll
        for (int a = 0; a < TT; ++a)
#pragma unroll
            for (int c = 0; c < TT; ++c) acc[a * TT + c] += yv[a] * zv[c];
    }
}
template <int TT>
__device__ __forceinline__ void gram_store(int np, const double* acc, double* M, int ld) {
    const int ng = np / TT;
    if ((int)threadIdx.x >= ng * ng) return;
    const int r0 = threadIdx.x / ng * TT, c0 = threadIdx.x % ng * TT;
#pragma unroll
    for (int a = 0; a < TT; ++a)
#pragma unroll
        for (int c = 0; c < TT; ++c) M[(r0 + a) * ld + c0 + c] = acc[a * TT + c];
}

// ---- twisted form: complex matrices are planar (real columns, then imaginary ones)

// Element (j, i) of the inverse G of a spin block: real part at p[j sj + i si],
// imaginary part `im` further on.
struct GView {
    const double* p;
    int sj, si, im;
    __device__ __forceinline__ double2 at(int j, int i) const {
        const double* q = p + (size_t)j * sj + (size_t)i * si;
        return make_double2(q[0], q[im]);
    }
};

// Z[r][i] = sum_j C[r][j] G[j][i] for `rows` rows of C, 4 x 2 complex outputs a thread.
__device__ __forceinline__ void tw_z(int rows, int n, int np, const double* __restrict__ C, const GView& G, double* out,
                                     int ld) {
    const int ncg = np / 2, tasks = (rows + 3) / 4 * ncg;
    for (int task = threadIdx.x; task < tasks; task += kThreads) {
        const int r0 = task / ncg * 4, c0 = task % ncg * 2;
        const int i0 = c0 < n ? c0 : n - 1, i1 = c0 + 1 < n ? c0 + 1 : n - 1;
        const double* ar[4];
#pragma unroll
        for (int a = 0; a < 4; ++a) ar[a] = C + (size_t)(r0 + a < rows ? r0 + a : rows - 1) * n;
        double acc[4][4] = {};
        for (int j = 0; j < n; ++j) {
            const double2 g0 = G.at(j, i0), g1 = G.at(j, i1);
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const double c = ar[a][j];
                acc[a][0] += c * g0.x; acc[a][1] += c * g1.x; acc[a][2] += c * g0.y; acc[a][3] += c * g1.y;
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
            if (r0 + a < rows) {
                double* o = out + (size_t)(r0 + a) * ld + c0;
                o[0] = acc[a][0]; o[1] = acc[a][1]; o[np] = acc[a][2]; o[np + 1] = acc[a][3];
            }
    }
}

// Y[r][j] += sum_{b < rows} y[b][r] C[b][j], r over the 2 np planar columns of y
// (real, then imaginary part of electron i), 2 x 4 outputs a thread.
__device__ __forceinline__ void tw_y(int rows, int n, int np, const double* y, int ld, const double* __restrict__ C,
                                     double* Y, int ldy) {
    const int ncg = np / 4, tasks = np * ncg;
    for (int task = threadIdx.x; task < tasks; task += kThreads) {
        const int r0 = task / ncg * 2, j0 = task % ncg * 4;
        double acc[2][4] = {};
        for (int b = 0; b < rows; ++b) {
            const double y0 = y[b * ld + r0], y1 = y[b * ld + r0 + 1];
            const double* c = C + (size_t)b * n;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const double cv = c[j0 + k < n ? j0 + k : n - 1];
                acc[0][k] += y0 * cv;
                acc[1][k] += y1 * cv;
            }
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            Y[(size_t)r0 * ldy + j0 + k] += acc[0][k];
            Y[(size_t)(r0 + 1) * ldy + j0 + k] += acc[1][k];
        }
    }
}

// T[i][c] = sum_j Y[i][j] G[j][c], 2 x 2 complex outputs a thread.
__device__ __forceinline__ void tw_yg(int n, int np, const double* Y, int ldy, const GView& G, double* T, int ld) {
    const int ng = np / 2;
    for (int task = threadIdx.x; task < ng * ng; task += kThreads) {
        const int i0 = task / ng * 2, c0 = task % ng * 2;
        const int ca = c0 < n ? c0 : n - 1, cb = c0 + 1 < n ? c0 + 1 : n - 1;
        double2 acc[2][2] = {};
        for (int j = 0; j < n; ++j) {
            const double2 g[2] = {G.at(j, ca), G.at(j, cb)};
#pragma unroll
            for (int a = 0; a < 2; ++a) {
                const double re = Y[(size_t)(i0 + a) * ldy + j], im = Y[(size_t)(np + i0 + a) * ldy + j];
#pragma unroll
                for (int c = 0; c < 2; ++c) {
                    acc[a][c].x += re * g[c].x - im * g[c].y;
                    acc[a][c].y += re * g[c].y + im * g[c].x;
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                T[(size_t)(i0 + a) * ld + c0 + c] = acc[a][c].x;
                T[(size_t)(i0 + a) * ld + np + c0 + c] = acc[a][c].y;
            }
    }
}

// K[j][c] = sum_i G[j][i] T[i][c], 2 x 2 complex outputs a thread.
__device__ __forceinline__ void tw_gt(int n, int np, const GView& G, const double* T, int ld, double* K) {
    const int ng = np / 2;
    for (int task = threadIdx.x; task < ng * ng; task += kThreads) {
        const int j0 = task / ng * 2, c0 = task % ng * 2;
        const int ja = j0 < n ? j0 : n - 1, jb = j0 + 1 < n ? j0 + 1 : n - 1;
        double2 acc[2][2] = {};
        for (int i = 0; i < n; ++i) {
            const double2 g[2] = {G.at(ja, i), G.at(jb, i)};
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                const double re = T[(size_t)i * ld + c0 + c], im = T[(size_t)i * ld + np + c0 + c];
#pragma unroll
                for (int a = 0; a < 2; ++a) {
                    acc[a][c].x += g[a].x * re - g[a].y * im;
                    acc[a][c].y += g[a].x * im + g[a].y * re;
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 2; ++a)
#pragma unroll
            for (int c = 0; c < 2; ++c) {
                K[(size_t)(j0 + a) * ld + c0 + c] = acc[a][c].x;
                K[(size_t)(j0 + a) * ld + np + c0 + c] = acc[a][c].y;
            }
    }
}

// e-e-n-n Jastrow orbital chi_a(r_i) = exp(-zeta |d|^2) with its gradient, Hessian,
// Laplacian and gradient of the Laplacian in the electron coordinate.
__device__ __forceinline__ double jas34(const double* ei, const double* pa, double ell, double zeta, double k2,
                                        RadialDerivs<double>& rd) {
    const Geo g = geometry(ei, pa, ell);
    const double e = qexp(-zeta * g.t);
    radial_chain(g.p, g.q, -zeta * e, zeta * zeta * e, -zeta * zeta * zeta * e, k2, rd);
    return e;
}

// TM: outputs a side per thread of the real form's np x np products (np / TM squared
// <= 256 threads); 0: the twisted form (its shared memory allows one CTA an SM).
template <int TM>
__global__ void __launch_bounds__(kThreads, TM ? 2 : 1) measure64_kernel(SysView<double> s, TwistView tv, int mmax, int tb,
                                                                int ntask,
                                                                const int4* __restrict__ ktask,
                                                                const double* __restrict__ kxyz,
                                                                const double* __restrict__ X,
                                                                const double* __restrict__ Gt,
                                                                const double* __restrict__ logdet,
                                                                double* __restrict__ acc, double* __restrict__ out_el,
                                                                double* __restrict__ out_lnpsi,
                                                                double* __restrict__ out_dl,
                                                                double* __restrict__ out_de) {
    extern __shared__ __align__(16) unsigned char sm[];
    const int N = s.N, n = s.n, Gn = s.G, B = s.B, nk = s.nk, np = s.np;
    const bool j34 = s.fj != nullptr;
    const M64Layout lay(N, n, np, nk, mmax, TM == 0, j34, tb);
    double* xs = (double*)(sm + lay.xs);
    double* et = (double*)(sm + lay.et);
    double* gU = (double*)(sm + lay.gU);
    double* lU = (double*)(sm + lay.lU);
    double* Ui = (double*)(sm + lay.Ui);
    double* gi = (double*)(sm + lay.gi);
    double* vvs = (double*)(sm + lay.vv);
    double* li = (double*)(sm + lay.li);
    double* f_dl = (double*)(sm + lay.facc);
    double* f_de = f_dl + 3 * N;
    double* f_dv = f_de + 3 * N;
    double2* rhot = (double2*)(sm + lay.rhot);
    double* red = (double*)(sm + lay.red);
    double* part = (double*)(sm + lay.part);
    double* uni = (double*)(sm + lay.uni);

    const int w = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const double L = s.L, iL = s.iL, ell = s.ell, bee = s.b_ee, bep = s.b_ep, Zj = s.Zj;
    const double twopiL = 2.0 * kPi * iL, k2 = twopiL * twopiL;

    // ---- positions and their (sin, cos)(pi x / L)
    for (int idx = tid; idx < 3 * N; idx += kThreads) {
        const double x = X[(size_t)w * 3 * N + idx];
        xs[idx] = x;
        double sn, cs;
        sincospi(x * iL, &sn, &cs);
        et[6 * (idx / 3) + idx % 3] = sn;
        et[6 * (idx / 3) + 3 + idx % 3] = cs;
    }
    for (int idx = tid; idx < 9 * N; idx += kThreads) f_dl[idx] = 0.0;
    __syncthreads();

    // ---- Jastrow gradient / Laplacian per electron and U, the partner range cut
    // into nparts slices so that every thread works, the slices summed in order.  An
    // e-e pair is evaluated once: electron i with i + d (mod N), d = 1..N/2 (d = N/2
    // only for i < N/2); at each distance every electron of a slice is one pair's
    // partner, whose share goes to its slot of the slice (a barrier per distance).
    const int nparts = kThreads >= N ? kThreads / N : 1, half = N / 2;
    double* partner = part + (size_t)5 * nparts * N;      // [nparts][N][4]
    for (int idx = tid; idx < 4 * nparts * N; idx += kThreads) partner[idx] = 0.0;
    __syncthreads();
    {
        const int i = tid % N, pi = tid / N;
        const bool on = pi < nparts;
        const int d0 = 1 + (half * pi) / nparts, d1 = 1 + (half * (pi + 1)) / nparts;
        const int j0 = (N * pi) / nparts, j1 = (N * (pi + 1)) / nparts, steps = (half + nparts - 1) / nparts;
        double g[3] = {0, 0, 0}, lp = 0, ui = 0;
        double ei[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) ei[c] = et[6 * i + c];
        for (int q = 0; q < steps; ++q) {
            const int d = d0 + q;
            if (on && d < d1 && !(2 * d == N && i >= half)) {
                const int j = i + d < N ? i + d : i + d - N;
                const Geo o = geometry(ei, et + 6 * j, ell);
                double u, c2, c4;
                pade_factors(o.t, bee, 0.5, u, c2, c4);
                const double pp = o.p[0] * o.p[0] + o.p[1] * o.p[1] + o.p[2] * o.p[2];
                const double lv = c4 * pp + c2 * (o.q[0] + o.q[1] + o.q[2]);
                double* pj = partner + 4 * ((size_t)pi * N + j);
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) {
                    const double gm = c2 * o.p[mu];       // odd under the exchange of the pair
                    g[mu] += gm;
                    pj[mu] -= gm;
                }
                lp += lv;
                pj[3] += lv;
                ui += u;
            }
            __syncthreads();
        }
        for (int a = j0; on && a < j1; ++a) {
            const Geo o = geometry(ei, s.ptrig + 6 * a, ell);
            double u, c2, c4;
            pade_factors(o.t, bep, -Zj, u, c2, c4);
            const double pp = o.p[0] * o.p[0] + o.p[1] * o.p[1] + o.p[2] * o.p[2];
            lp += c4 * pp + c2 * (o.q[0] + o.q[1] + o.q[2]);
#pragma unroll
            for (int mu = 0; mu < 3; ++mu) g[mu] += c2 * o.p[mu];
            ui += u;
        }
        if (on) {
            double* o = part + 5 * ((size_t)pi * N + i);
            const double* pj = partner + 4 * ((size_t)pi * N + i);
            o[0] = g[0] + pj[0]; o[1] = g[1] + pj[1]; o[2] = g[2] + pj[2]; o[3] = lp + pj[3]; o[4] = ui;
        }
    }
    __syncthreads();
    for (int i = tid; i < N; i += kThreads) {
        double v[5] = {0, 0, 0, 0, 0};
        for (int pi = 0; pi < nparts; ++pi)
#pragma unroll
            for (int c = 0; c < 5; ++c) v[c] += part[((size_t)pi * N + i) * 5 + c];
        gU[3 * i] = v[0]; gU[3 * i + 1] = v[1]; gU[3 * i + 2] = v[2];
        lU[i] = v[3]; Ui[i] = v[4];
    }
    __syncthreads();

    // ---- e-e-n-n Jastrow term:
    //   U34 = sum_{i<j} chi_i^T F chi_j = 1/2 sum_i chi_i . w_i,  w_i = F (c - chi_i),  c = sum_j chi_j,
    //   grad_i U34 = sum_a grad chi_a(r_i) w_ia,  lap_i U34 = sum_a lap chi_a(r_i) w_ia.
    // c and S_a = sum_j grad chi_a(r_j) are formed again for the force terms below
    // (the orbital products use the work space in between).
    double* j34c = uni;              // [N]
    double* j34S = j34c + N;         // [N][3]
    double* st = j34S + 3 * N + (size_t)warp * 5 * N;   // per warp: c - chi_i [N], grad chi_i [N][3], lap chi_i [N]
    double* j34f = j34S + 3 * N + (size_t)kWarps * 5 * N;   // [6][kWarps][N] force terms of the warps' electrons
    const double zj = s.zeta_j;
    auto j34_sums = [&]() {
        for (int a = tid; a < N; a += kThreads) {
            double c = 0, g[3] = {0, 0, 0};
            for (int j = 0; j < N; ++j) {
                RadialDerivs<double> rd;
                c += jas34(et + 6 * j, s.ptrig + 6 * a, ell, zj, k2, rd);
                for (int mu = 0; mu < 3; ++mu) g[mu] += rd.g[mu];
            }
            j34c[a] = c;
            for (int mu = 0; mu < 3; ++mu) j34S[3 * a + mu] = g[mu];
        }
        __syncthreads();
    };
    if (j34) {
        j34_sums();
        for (int i = warp; i < N; i += kWarps) {
            for (int a = lane; a < N; a += 32) {
                RadialDerivs<double> rd;
                st[a] = j34c[a] - jas34(et + 6 * i, s.ptrig + 6 * a, ell, zj, k2, rd);
            }
            __syncwarp();
            double g[3] = {0, 0, 0}, l = 0, u = 0;
            for (int a = lane; a < N; a += 32) {
                RadialDerivs<double> rd;
                const double chi = jas34(et + 6 * i, s.ptrig + 6 * a, ell, zj, k2, rd);
                const double* fa = s.fj + a;   // column a = row a (f symmetric): coalesced over lanes
                double wa = 0;
                for (int b = 0; b < N; ++b) wa += fa[(size_t)b * N] * st[b];
                for (int mu = 0; mu < 3; ++mu) g[mu] += rd.g[mu] * wa;
                l += rd.lap * wa;
                u += chi * wa;
            }
            for (int mu = 0; mu < 3; ++mu) g[mu] = warp_sum(g[mu]);
            l = warp_sum(l);
            u = warp_sum(u);
            if (lane == 0) {
                for (int mu = 0; mu < 3; ++mu) gU[3 * i + mu] += g[mu];
                lU[i] += l;
                Ui[i] += 0.5 * u;
            }
            __syncwarp();
        }
        __syncthreads();
    }

    // ---- orbital terms, one spin block at a time
    const int seg = np < 32 ? np : 32, apw = 32 / seg;   // lanes per nucleus, nuclei per warp
    const int sub = lane / seg, sl = lane - sub * seg;
    // a nucleus' sums over its lanes: v = dl (3), de (3)
    auto add_forces = [&](double v[8], int a, bool on) {
        if (seg == 32) {
            const double x = warp_sum8(v, lane);
            const int q = lane >> 2;
            if ((lane & 3) == 0 && q < 6) (q < 3 ? f_dl : f_de)[3 * a + q % 3] += x;
        } else {
            seg_sum(v, 6, seg);
            if (sl == 0 && on)
#pragma unroll
                for (int mu = 0; mu < 3; ++mu) { f_dl[3 * a + mu] += v[mu]; f_de[3 * a + mu] += v[3 + mu]; }
        }
    };
    // g_i, l_i of spin block sp from the lanes' sums: the segments of a warp, then the warps in order
    auto gather_gl = [&](double ga[2][4], int sp) {
        for (int o = seg; o < 32; o <<= 1)
#pragma unroll
            for (int c = 0; c < 4; ++c) ga[0][c] += __shfl_xor_sync(0xffffffffu, ga[0][c], o);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int il = sl + 32 * h;
            if (sub == 0 && il < n)
#pragma unroll
                for (int c = 0; c < 4; ++c) part[((size_t)warp * n + il) * 4 + c] = ga[h][c];
        }
        __syncthreads();
        for (int idx = tid; idx < 4 * n; idx += kThreads) {
            double v = 0;
            for (int q = 0; q < kWarps; ++q) v += part[(size_t)q * n * 4 + idx];
            const int i = sp * n + (idx >> 2), c = idx & 3;
            if (c < 3) gi[3 * i + c] = v;
            else li[i] = v;
        }
    };
    if constexpr (TM != 0) {
        const int ld = np + 2;
        double* Gm = uni;                         // G[j][i]
        double* Mm = Gm + (size_t)np * ld;        // M[i'][i]
        double* Zs = Mm + (size_t)np * ld;        // [tb][ld] Z
        double* Cs = Zs + (size_t)tb * ld;        // [tb][ld] 2 zeta chi
        double* Ys = Cs + (size_t)tb * ld;        // [tb][ld] y, then P
        const bool whole = tb >= B;
        for (int sp = 0; sp < 2; ++sp) {
            const double* Gsp = Gt + ((size_t)w * 2 + sp) * n * n;
            for (int idx = tid; idx < np * np; idx += kThreads) {
                const int i = idx / np, j = idx - i * np;
                Gm[j * ld + i] = (i < n && j < n) ? Gsp[i * n + j] : 0.0;
            }
            double macc[TM * TM] = {};
            double ga[2][4] = {};                 // g_i, l_i of this lane's electrons (two where n > 32)
            __syncthreads();
            for (int pass = 0; pass < 2; ++pass) {
                for (int b0 = 0; b0 < B; b0 += tb) {
                    const int rows = B - b0 < tb ? B - b0 : tb, a0 = b0 / Gn, na = rows / Gn;
                    if (pass == 0 || !whole) {
                        product_any(rows, np, n, s.C + (size_t)b0 * n, n, rows, Gm, ld, Zs, ld);
                        __syncthreads();
                    }
                    if (pass == 1) {
                        product_any(rows, np, n, Zs, ld, rows, Mm, ld, Ys, ld);
                        __syncthreads();
                    }
                    // basis pass: a warp (or a segment of it) per nucleus, lanes over the spin's electrons
                    for (int ab = warp * apw; ab < na; ab += kWarps * apw) {
                        const int al = ab + sub, a = a0 + al;
                        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // dl, de
                        if (al < na) {
                            double pa[6];
#pragma unroll
                            for (int c = 0; c < 6; ++c) pa[c] = s.ptrig[6 * a + c];
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const int il = sl + 32 * h;
                                if (il >= n) continue;
                                const int i = sp * n + il;
                                const Geo o = geometry(et + 6 * i, pa, ell);
                                const int base = al * Gn * ld + il;
                                if (pass == 0) {
                                    const double* gu = gU + 3 * i;
                                    const double pp = o.p[0] * o.p[0] + o.p[1] * o.p[1] + o.p[2] * o.p[2];
                                    const double sq = o.q[0] + o.q[1] + o.q[2];
                                    const double pg = o.p[0] * gu[0] + o.p[1] * gu[1] + o.p[2] * gu[2];
                                    const double sp2 = fma(2.0, pg, sq), pp2 = 2.0 * pp;
                                    double s1 = 0, s2 = 0, s3 = 0;   // sum_g Z zeta^q chi
                                    for (int g = 0; g < Gn; ++g) {
                                        const double z = s.zeta[g];
                                        const double w1 = z * qexp(-z * o.t), w2 = z * w1;
                                        const double Z = Zs[base + g * ld];
                                        Cs[base + g * ld] = 2.0 * w1;
                                        Ys[base + g * ld] = fma(w1, sp2, -(w2 * pp2));
                                        s1 = fma(Z, w1, s1); s2 = fma(Z, w2, s2); s3 = fma(Z, z * w2, s3);
                                    }
                                    s1 = -2.0 * s1; s2 *= 4.0;       // 2 s1 and 4 s2 of the header; s3 = -s3
                                    const double c0 = fma(s2, pg, fma(-4.0 * s3, pp, fma(0.5 * s2, sq, -0.5 * k2 * s1)));
                                    ga[h][3] += fma(s2, pp, s1 * sq);
#pragma unroll
                                    for (int mu = 0; mu < 3; ++mu) {
                                        const double gr = s1 * o.p[mu];
                                        ga[h][mu] += gr;
                                        v[mu] -= gr;
                                        v[3 + mu] += fma(o.p[mu], fma(s2, o.q[mu], c0), s1 * (o.q[mu] * gu[mu]));
                                    }
                                } else {
                                    double pc = 0;                   // -sum_g P_bi 2 zeta chi
                                    if (whole) {
                                        for (int g = 0; g < Gn; ++g) pc = fma(Ys[base + g * ld], Cs[base + g * ld], pc);
                                    } else {
                                        for (int g = 0; g < Gn; ++g) {
                                            const double z = s.zeta[g];
                                            pc = fma(Ys[base + g * ld], 2.0 * z * qexp(-z * o.t), pc);
                                        }
                                    }
#pragma unroll
                                    for (int mu = 0; mu < 3; ++mu) v[3 + mu] -= pc * o.p[mu];
                                }
                            }
                        }
                        add_forces(v, a, al < na);
                    }
                    __syncthreads();
                    if (pass == 0) {
                        gram_acc<TM>(rows, np, Ys, Zs, ld, macc);
                        if (!whole) __syncthreads();
                    }
                }
                if (pass == 0) {
                    gram_store<TM>(np, macc, Mm, ld);
                    gather_gl(ga, sp);
                }
            }
            __syncthreads();
        }
    } else {
        const int ld2 = 2 * np + 2, ldy = np + 2, M = tv.M, t = w / tv.Wk;
        const size_t sq = M64Layout::square2(np);
        double* Gs = uni;                                   // G (np <= 32)
        double* YK = Gs + (np <= 32 ? sq : 0);              // Y [2 np][ldy], then K [np][ld2]
        double* tile = YK + sq;                             // [tb][ld2]: Z, overwritten by y; P.  T [np][ld2] in between
        const double2* ph = tv.ph + (size_t)t * 3 * (2 * M + 1);
        const double* th = tv.theta + 3 * t;
        __shared__ int images[8][2];                        // per Gaussian: near and far images (n_gauss <= 8)
        if (tid < Gn) {
            images[tid][0] = bloch_near(s.zeta[tid], L, M);
            images[tid][1] = bloch_far(s.zeta[tid], L, M);
        }
        for (int sp = 0; sp < 2; ++sp) {
            const double sg = sp == 0 ? 1.0 : -1.0;
            const double2* Gsp = (const double2*)Gt + ((size_t)w * 2 + sp) * n * n;   // G^T[i][j] = G[j][i]
            GView G{(const double*)Gsp, 2, 2 * n, 1};
            if (np <= 32) {
                for (int idx = tid; idx < n * n; idx += kThreads) {
                    const int i = idx / n, j = idx - i * n;
                    const double2 g = Gsp[idx];
                    Gs[(size_t)j * ld2 + i] = g.x;
                    Gs[(size_t)j * ld2 + np + i] = g.y;
                }
                G = GView{Gs, ld2, 1, np};
            }
            for (int idx = tid; idx < 2 * np * ldy; idx += kThreads) YK[idx] = 0.0;
            double ga[2][4] = {};
            __syncthreads();
            for (int pass = 0; pass < 2; ++pass) {
                for (int b0 = 0; b0 < B; b0 += tb) {
                    const int rows = B - b0 < tb ? B - b0 : tb, a0 = b0 / Gn, na = rows / Gn;
                    const double* Ct = s.C + (size_t)b0 * n;
                    if (pass == 0) tw_z(rows, n, np, Ct, G, tile, ld2);
                    else product_any(rows, 2 * np, n, Ct, n, rows, YK, ld2, tile, ld2);    // P = C K
                    __syncthreads();
                    for (int ab = warp * apw; ab < na; ab += kWarps * apw) {
                        const int al = ab + sub, a = a0 + al;
                        double v[8] = {0, 0, 0, 0, 0, 0, 0, 0};   // dl, de
                        if (al < na) {
#pragma unroll 1
                            for (int h = 0; h < 2; ++h) {
                                const int il = sl + 32 * h;
                                if (il >= n) continue;
                                const int i = sp * n + il;
                                double d0[3];
                                const double2 P = bloch_min_image(xs + 3 * i, s.R + 3 * a, L, iL, M, ph, th, sg, d0);
                                double* zt = tile + (size_t)al * Gn * ld2 + il;
                                const double* gu = gU + 3 * i;
#pragma unroll 1
                                for (int g = 0; g < Gn; ++g, zt += ld2) {
                                    const double z = s.zeta[g];
                                    const int near = images[g][0], far = images[g][1];
                                    const double2 zp = cmul(make_double2(zt[0], zt[np]), P);
                                    if (pass == 0) {
                                        double2 sx[4], sy[4], sz[4];
                                        bloch_axis<3>(d0[0], z, L, near, far, M, ph, sg, sx);
                                        bloch_axis<3>(d0[1], z, L, near, far, M, ph + (2 * M + 1), sg, sy);
                                        bloch_axis<3>(d0[2], z, L, near, far, M, ph + 2 * (2 * M + 1), sg, sz);
                                        const double2 tx = caxpy(gu[0], sx[1], 0.5, sx[2]), ty = caxpy(gu[1], sy[1], 0.5, sy[2]),
                                                      tz = caxpy(gu[2], sz[1], 0.5, sz[2]);
                                        const double2 ux = caxpy(gu[0], sx[2], 0.5, sx[3]), uy = caxpy(gu[1], sy[2], 0.5, sy[3]),
                                                      uz = caxpy(gu[2], sz[2], 0.5, sz[3]);
                                        const double2 yz = cmul(sy[0], sz[0]), xz = cmul(sx[0], sz[0]), xy = cmul(sx[0], sy[0]);
                                        const double2 ayz = cadd(cmul(ty, sz[0]), cmul(sy[0], tz)),
                                                      axz = cadd(cmul(tx, sz[0]), cmul(sx[0], tz)),
                                                      axy = cadd(cmul(tx, sy[0]), cmul(sx[0], ty));
                                        const double2 y = cmul(P, cadd(cmul(tx, yz), cmul(sx[0], ayz)));
                                        zt[0] = -y.x;
                                        zt[np] = -y.y;
                                        const double gr[3] = {cre(zp, cmul(sx[1], yz)), cre(zp, cmul(sy[1], xz)),
                                                              cre(zp, cmul(sz[1], xy))};
                                        ga[h][3] += cre(zp, cadd(cadd(cmul(sx[2], yz), cmul(sy[2], xz)), cmul(sz[2], xy)));
                                        v[3] += cre(zp, cadd(cmul(ux, yz), cmul(sx[1], ayz)));
                                        v[4] += cre(zp, cadd(cmul(uy, xz), cmul(sy[1], axz)));
                                        v[5] += cre(zp, cadd(cmul(uz, xy), cmul(sz[1], axy)));
#pragma unroll
                                        for (int mu = 0; mu < 3; ++mu) { ga[h][mu] += gr[mu]; v[mu] -= gr[mu]; }
                                    } else {
                                        double2 sx[2], sy[2], sz[2];
                                        bloch_axis<1>(d0[0], z, L, near, far, M, ph, sg, sx);
                                        bloch_axis<1>(d0[1], z, L, near, far, M, ph + (2 * M + 1), sg, sy);
                                        bloch_axis<1>(d0[2], z, L, near, far, M, ph + 2 * (2 * M + 1), sg, sz);
                                        const double2 px = cmul(zp, sx[0]);
                                        v[3] += cre(cmul(zp, sx[1]), cmul(sy[0], sz[0]));
                                        v[4] += cre(cmul(px, sy[1]), sz[0]);
                                        v[5] += cre(cmul(px, sy[0]), sz[1]);
                                    }
                                }
                            }
                        }
                        add_forces(v, a, al < na);
                    }
                    __syncthreads();
                    if (pass == 0) {
                        tw_y(rows, n, np, tile, ld2, Ct, YK, ldy);
                        __syncthreads();
                    }
                }
                if (pass == 0) {
                    tw_yg(n, np, YK, ldy, G, tile, ld2);   // T = Y G
                    __syncthreads();
                    tw_gt(n, np, G, tile, ld2, YK);        // K = G T over Y
                    gather_gl(ga, sp);                     // (its barrier ends the reads of T too)
                }
            }
            __syncthreads();
        }
    }

    // ---- kinetic energy and U
    double kin_p = 0.0, u_p = 0.0;
    for (int i = tid; i < N; i += kThreads) {
        double g2 = 0, t2 = 0;
#pragma unroll
        for (int mu = 0; mu < 3; ++mu) {
            const double g = gi[3 * i + mu], t = g + gU[3 * i + mu];
            g2 += g * g; t2 += t * t;
            vvs[3 * i + mu] = t;     // grad_i ln psi, for the e-n pair terms
        }
        kin_p += li[i] - g2 + lU[i] + t2;
        u_p += Ui[i];
    }
    const double kin = block_sum(kin_p, red);
    const double Utot = block_sum(u_p, red + 32);

    // ---- e-e-n-n terms of d ln psi / dR_a and dE_L / dR_a.  With s_a^(i) = S_a -
    // grad chi_a(r_i), v_ia = sum_b grad chi_b(r_i) f_ba, lam_ia = sum_b lap chi_b(r_i) f_ba
    // and vv_i = g_i + grad_i U:
    //   dlnpsi/dR_a += -sum_i grad chi_a(r_i) w_ia
    //   dE_L/dR_a   += sum_i [ 1/2 (grad lap chi_a(r_i) w_ia + lam_ia s_a^(i))
    //                          + (Hess chi_a(r_i) vv_i) w_ia + (vv_i . v_ia) s_a^(i) ]
    // (the R_a-derivative of -1/2 sum_i [lap_i U34 + 2 vv_i . grad_i U34]).
    if (j34) {
        // a warp adds its electrons' terms up in its own slots, the warps are added in order
        for (int idx = tid; idx < 6 * kWarps * N; idx += kThreads) j34f[idx] = 0.0;
        j34_sums();
        for (int i = warp; i < N; i += kWarps) {
            for (int a = lane; a < N; a += 32) {
                RadialDerivs<double> rd;
                st[a] = j34c[a] - jas34(et + 6 * i, s.ptrig + 6 * a, ell, zj, k2, rd);
                for (int mu = 0; mu < 3; ++mu) st[N + 3 * a + mu] = rd.g[mu];
                st[4 * N + a] = rd.lap;
            }
            __syncwarp();
            double vv[3];
            for (int mu = 0; mu < 3; ++mu) vv[mu] = vvs[3 * i + mu];
            for (int a = lane; a < N; a += 32) {
                RadialDerivs<double> rd;
                jas34(et + 6 * i, s.ptrig + 6 * a, ell, zj, k2, rd);
                const double* fa = s.fj + a;   // column a = row a (f symmetric): coalesced over lanes
                double wa = 0, v[3] = {0, 0, 0}, lam = 0;
                for (int b = 0; b < N; ++b) {
                    const double f = fa[(size_t)b * N];
                    wa += f * st[b];
                    for (int mu = 0; mu < 3; ++mu) v[mu] += st[N + 3 * b + mu] * f;
                    lam += st[4 * N + b] * f;
                }
                double hv[3];
                hess_mul(rd.h, vv, hv);
                const double vvv = vv[0] * v[0] + vv[1] * v[1] + vv[2] * v[2];
                double* o = j34f + (size_t)warp * N + a;
                for (int mu = 0; mu < 3; ++mu) {
                    const double sa = j34S[3 * a + mu] - rd.g[mu];
                    o[mu * kWarps * N] -= rd.g[mu] * wa;
                    o[(3 + mu) * kWarps * N] += 0.5 * (rd.tl[mu] * wa + lam * sa) + hv[mu] * wa + vvv * sa;
                }
            }
            __syncwarp();
        }
        __syncthreads();
        for (int idx = tid; idx < 6 * N; idx += kThreads) {
            const int c = idx / N, a = idx - c * N;
            double t = 0;
            for (int q = 0; q < kWarps; ++q) t += j34f[(size_t)(c * kWarps + q) * N + a];
            (c < 3 ? f_dl : f_de)[3 * a + c % 3] += t;
        }
        __syncthreads();
    }

    // ---- electron-electron real-space Ewald: balanced cyclic pairing, electron i
    // with i + d (mod N), d = 1..N/2 (d = N/2 only for i < N/2), in nparts slices
    const EwTable ewt{s.ewt, s.ew_h, s.ew_ih, L, iL, L * L};
    double vee_p = 0.0;
    for (int tt = tid; tt < nparts * N; tt += kThreads) {
        const int i = tt % N, pi = tt / N;
        const int d0 = 1 + (half * pi) / nparts, d1 = 1 + (half * (pi + 1)) / nparts;
        double v = 0;
        for (int d = d0; d < d1; ++d) {
            if (2 * d == N && i >= half) continue;
            const int j = i + d < N ? i + d : i + d - N;
            const double dx = xs[3 * i] - xs[3 * j], dy = xs[3 * i + 1] - xs[3 * j + 1],
                         dz = xs[3 * i + 2] - xs[3 * j + 2];
            v += ewt.t ? ewald_table<false>(dx, dy, dz, ewt, nullptr) : ewald_real<double>(dx, dy, dz, L, s.kappa, nullptr);
        }
        vee_p += v;
    }
    // ---- electron-proton pairs: the real-space Ewald energy and its R-gradient
    // (Hellmann-Feynman) together with the e-n Jastrow terms of d ln psi/dR and
    // dE_L/dR.  A warp (N < 32: a segment of it) per proton, lanes over electrons.
    double vep_p = 0.0;
    {
        int seg = 32;
        while (seg > 4 && seg / 2 >= N) seg >>= 1;
        const int apw = 32 / seg, sub = lane / seg, sl = lane - sub * seg;
        for (int ab = warp * apw; ab < N; ab += kWarps * apw) {
            const int a = ab + sub;
            double v[8] = {0, 0, 0, 0, 0, 0, 0, 0}, e0 = 0, e1 = 0;   // energy, gradient, dl, de x | de y, de z
            if (a < N) {
                double pa[6], ra[3];
#pragma unroll
                for (int c = 0; c < 6; ++c) pa[c] = s.ptrig[6 * a + c];
#pragma unroll
                for (int c = 0; c < 3; ++c) ra[c] = s.R[3 * a + c];
                for (int i = sl; i < N; i += seg) {
                    const Geo o = geometry(et + 6 * i, pa, ell);
                    const double* vv = vvs + 3 * i;
                    double c2, c4, c8, pg[3];
                    pade_factors3(o.t, bep, -Zj, c2, c4, c8);
                    const double pp = o.p[0] * o.p[0] + o.p[1] * o.p[1] + o.p[2] * o.p[2];
                    const double pv = o.p[0] * vv[0] + o.p[1] * vv[1] + o.p[2] * vv[2];
                    // H v + 1/2 grad lap: p (c4 p.v + 1/2 (c8 |p|^2 + c4 sum q - k2 c2) + c4 q) + c2 q o v
                    const double c0 = fma(c4, pv, 0.5 * fma(c8, pp, fma(c4, o.q[0] + o.q[1] + o.q[2], -k2 * c2)));
                    double de[3];
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) {
                        v[4 + mu] -= c2 * o.p[mu];
                        de[mu] = fma(o.p[mu], fma(c4, o.q[mu], c0), c2 * (o.q[mu] * vv[mu]));
                    }
                    v[7] += de[0]; e0 += de[1]; e1 += de[2];
                    const double dx = xs[3 * i] - ra[0], dy = xs[3 * i + 1] - ra[1], dz = xs[3 * i + 2] - ra[2];
                    v[0] += ewt.t ? ewald_table<true>(dx, dy, dz, ewt, pg) : ewald_real<double>(dx, dy, dz, L, s.kappa, pg);
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) v[1 + mu] += pg[mu];
                }
            }
            // proton charge 1
            if (seg == 32) {
                const double x = warp_sum8(v, lane);
                e0 = warp_sum(e0); e1 = warp_sum(e1);
                const int q = lane >> 2;
                if ((lane & 3) == 0) {
                    if (q == 0) vep_p -= x;
                    else if (q < 4) f_dv[3 * a + q - 1] += x;
                    else if (q < 7) f_dl[3 * a + q - 4] += x;
                    else { f_de[3 * a] += x; f_de[3 * a + 1] += e0; f_de[3 * a + 2] += e1; }
                }
            } else {
                seg_sum(v, 8, seg);
                seg_sum(&e0, 1, seg);
                seg_sum(&e1, 1, seg);
                if (sl == 0 && a < N) {
                    vep_p -= v[0];
#pragma unroll
                    for (int mu = 0; mu < 3; ++mu) { f_dv[3 * a + mu] += v[1 + mu]; f_dl[3 * a + mu] += v[4 + mu]; }
                    f_de[3 * a] += v[7]; f_de[3 * a + 1] += e0; f_de[3 * a + 2] += e1;
                }
            }
        }
    }
    // ---- reciprocal space: electron structure factor from per-electron phase
    // tables e^{i m theta}, m = 0..mmax (theta = 2 pi x / L by the double angle).
    // A task is two |m_z| of one (m_x, m_y): with ab the x y phase and c the z
    // phase, the four sums of ab.x c.x, ab.y c.y, ab.x c.y, ab.y c.x give rho at
    // both signs of m_z, 12 operations an electron for four vectors (32 before).
    __syncthreads();
    double2* etab = (double2*)uni;
    const int nm = mmax + 1;
    for (int idx = tid; idx < 3 * N; idx += kThreads) {
        const double sx = et[6 * (idx / 3) + idx % 3], cx = et[6 * (idx / 3) + 3 + idx % 3];
        const double sn = 2.0 * sx * cx, cs = fma(-2.0 * sx, sx, 1.0);
        double2* e = etab + (size_t)idx * nm;
        double2 cur = make_double2(1.0, 0.0);
        e[0] = cur;
        for (int m = 1; m <= mmax; ++m) {
            cur = make_double2(cur.x * cs - cur.y * sn, cur.x * sn + cur.y * cs);
            e[m] = cur;
        }
    }
    __syncthreads();
    double vrec_p = 0.0;
    for (int tk = tid; tk < ntask; tk += kThreads) {
        const int4 m = ktask[tk];                 // m_x >= 0, m_y, first |m_z|, index of (m_x, m_y, 0)
        const int my = m.y < 0 ? -m.y : m.y, z1 = m.z + 1 <= mmax ? m.z + 1 : mmax;
        const double sy = m.y < 0 ? -1.0 : 1.0;
        double q[2][4] = {};
        for (int i = 0; i < N; ++i) {
            const double2 a = etab[(3 * i) * nm + m.x], c0 = etab[(3 * i + 2) * nm + m.z], c1 = etab[(3 * i + 2) * nm + z1];
            double2 b = etab[(3 * i + 1) * nm + my];
            b.y *= sy;
            const double x = a.x * b.x - a.y * b.y, y = a.x * b.y + a.y * b.x;
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
                const double re = sg ? q[h][0] + q[h][1] : q[h][0] - q[h][1];
                const double im = sg ? q[h][3] - q[h][2] : q[h][3] + q[h][2];
                const double2 rp = s.rho_p[k];
                const double rr = rp.x - re, ri = rp.y - im;   // electrons carry -1
                const double kw = s.kw[k];
                rhot[k] = make_double2(2.0 * kw * rr, 2.0 * kw * ri);
                vrec_p += kw * (rr * rr + ri * ri);
            }
        }
    }
    __syncthreads();
    // ---- reciprocal-space force on the protons (warp per proton)
    for (int a = warp; a < N; a += kWarps) {
        double gx = 0, gy = 0, gz = 0;
#pragma unroll 4
        for (int k = lane; k < nk; k += 32) {
            const double2 e = s.eikR[(size_t)a * nk + k], rd = rhot[k];
            const double c = rd.y * e.x - rd.x * e.y;
            gx += c * kxyz[k]; gy += c * kxyz[nk + k]; gz += c * kxyz[2 * nk + k];
        }
        gx = warp_sum(gx); gy = warp_sum(gy); gz = warp_sum(gz);
        if (lane == 0) { f_dv[3 * a] += gx; f_dv[3 * a + 1] += gy; f_dv[3 * a + 2] += gz; }
    }
    const double vee = block_sum(vee_p, red);
    const double vep = block_sum(vep_p, red + 32);
    const double vrec = block_sum(vrec_p, red);
    __syncthreads();

    // ---- accumulate the sample
    const double V = vee + vep + vrec + s.vconst[0], EL = -0.5 * kin + V;
    const int N3 = 3 * N;
    double* aw = acc + (size_t)w * (3 + 9 * (size_t)N);
    bool bad = !isfinite(EL);
    for (int c = tid; c < N3; c += kThreads) {
        const double dl = f_dl[c], de = f_de[c] + f_dv[c] + s.dvpp[c];
        if (!isfinite(dl) || !isfinite(de)) bad = true;
        aw[3 + c] += dl;
        aw[3 + N3 + c] += EL * dl;
        aw[3 + 2 * N3 + c] += de;
        if (out_dl) { out_dl[(size_t)w * N3 + c] = dl; out_de[(size_t)w * N3 + c] = de; }
    }
    if (tid == 0) {
        aw[0] += 1.0; aw[1] += EL; aw[2] += EL * EL;
        if (s.vacc) s.vacc[w] += V;   // V_L, for the virial pressure
        if (out_el) { out_el[w] = EL; out_lnpsi[w] = logdet[2 * w] + logdet[2 * w + 1] + Utot; }
    }
    if (bad) raise_err(s.err, kErrNonfinite);
}

template <int TM>
void launch(const SysView<double>& s, const TwistView& tv, int tb, size_t smem, int ntask, const int4* ktask,
            const double* kxyz, const double* X, const double* Gt, const double* logdet, double* acc, double* out_el,
            double* out_lnpsi, double* out_dl, double* out_de, cudaStream_t st) {
    static bool set = false;
    if (!set) {
        cudaFuncSetAttribute(measure64_kernel<TM>, cudaFuncAttributeMaxDynamicSharedMemorySize, 226 * 1024);
        set = true;
    }
    measure64_kernel<TM><<<s.W, kThreads, smem, st>>>(s, tv, s.mmax, tb, ntask, ktask, kxyz, X, Gt, logdet, acc, out_el,
                                                      out_lnpsi, out_dl, out_de);
}

}  // namespace

void launch_measure64(const SysView<double>& s, const TwistView* tv, int ntask, const int4* ktask, const double* kxyz,
                      const double* X, const double* Gt, const double* logdet, double* acc, double* out_el,
                      double* out_lnpsi, double* out_dl, double* out_de, cudaStream_t st) {
    const bool j34 = s.fj != nullptr;
    const int tb = tile_rows(s.N, s.n, s.G, s.nk, s.mmax, tv != nullptr, j34);
    const size_t smem = M64Layout(s.N, s.n, s.np, s.nk, s.mmax, tv != nullptr, j34, tb).total;
    // np x np outputs over 256 threads: one, 2 x 2 or 4 x 4 each
    auto go = tv ? launch<0> : s.np <= 16 ? launch<1> : s.np <= 32 ? launch<2> : launch<4>;
    go(s, tv ? *tv : TwistView{}, tb, smem, ntask, ktask, kxyz, X, Gt, logdet, acc, out_el, out_lnpsi, out_dl, out_de, st);
}

}  // namespace qmc
