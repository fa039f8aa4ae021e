// k_invert.cu -- full FP64 inverse of every walker's two Slater blocks.
//
// A_s[i][j] = phi_j(r_i) for the n electrons of spin s.  In-place Gauss-Jordan
// with partial (row) pivoting (Golub & Van Loan sec. 3.4); row interchanges
// turn into column interchanges of the inverse, undone at the end.  Always
// FP64: this is the periodic recompute that resets the drift of the rank-1
// (Sherman-Morrison) updates of the sweep kernel.  Output: Gt[i][j] = (A^-1)_{j,i}
// in the working precision and ln|det A|.  The mixed form reaches FP64's accuracy
// with pairs of FP32 numbers above n = 16 (invert_pair_kernel).
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// Gauss-Jordan inverse of walker w's spin block sp by the whole CTA, in the
// FP64 work space sm (n (n + 1) + n doubles and n ints).
template <typename T>
__device__ void gj_invert(int N, int n, const T* __restrict__ Phi, T* __restrict__ Gt, double* __restrict__ logdet,
                          int* err, int w, int sp, double* sm) {
    const int ld = n + 1;
    double* M = sm;                      // [n][n+1]
    double* col = M + (size_t)n * ld;    // [n]
    int* perm = (int*)(col + n);         // [n]
    __shared__ int piv_row;
    __shared__ int singular;
    __shared__ double ipv_s;
    __shared__ int sgn;
    const int tid = threadIdx.x, nt = blockDim.x;
    const T* A = Phi + ((size_t)w * N + (size_t)sp * n) * n;
    for (int idx = tid; idx < n * n; idx += nt) M[(idx / n) * ld + idx % n] = (double)A[idx];
    if (tid == 0) { sgn = 1; singular = 0; }
    // ln|det| as mantissa product and exponent sum (one log at the end): the
    // FP64 pipe is the bound here, so no per-step log or per-thread division
    double mant = 1.0;
    int expo = 0;
    // rank-1 update: thread owns column jj of rows i0, i0 + istep, ... (no index division per element)
    const bool tiled = nt % n == 0;
    const int jj = tid % n, i0 = tid / n, istep = nt / n;
    __syncthreads();
    for (int k = 0; k < n; ++k) {
        if (tid < 32) {                      // argmax |M[i][k]|, i >= k (ties -> lowest row)
            // magnitudes compared as the bit patterns of |x| (monotonic for
            // finite doubles): integer work instead of FP64 compares
            unsigned long long best = 0ull; int bi = n;
            for (int i = k + tid; i < n; i += 32) {
                const unsigned long long v = (unsigned long long)__double_as_longlong(M[i * ld + k]) & 0x7FFFFFFFFFFFFFFFull;
                if (bi == n || v > best) { best = v; bi = i; }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
                const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
                if (oi < n && (bi == n || ob > best || (ob == best && oi < bi))) { best = ob; bi = oi; }
            }
            if (tid == 0) {
                piv_row = bi;
                perm[k] = bi;
                if (best == 0ull) singular = 1;
            }
        }
        __syncthreads();
        if (singular) break;
        const int p = piv_row;
        if (p != k) {
            for (int j = tid; j < n; j += nt) {
                const double t = M[k * ld + j];
                M[k * ld + j] = M[p * ld + j];
                M[p * ld + j] = t;
            }
            __syncthreads();
        }
        if (tid == 0) {
            const double pv = M[k * ld + k];
            int e1, e2;
            const double m1 = frexp(fabs(pv), &e1);
            mant = frexp(mant * m1, &e2);
            expo += e1 + e2;
            sgn *= (p != k ? -1 : 1) * (pv < 0 ? -1 : 1);
            ipv_s = 1.0 / pv;
        }
        for (int i = tid; i < n; i += nt) col[i] = (i == k) ? 0.0 : M[i * ld + k];
        __syncthreads();
        const double ipv = ipv_s;
        for (int j = tid; j < n; j += nt) M[k * ld + j] = (j == k ? 1.0 : M[k * ld + j]) * ipv;
        __syncthreads();
        if (tiled) {
            const double mkj = M[k * ld + jj];
            for (int i = i0; i < n; i += istep) {
                if (i == k) continue;
                const double base = (jj == k) ? 0.0 : M[i * ld + jj];
                M[i * ld + jj] = base - col[i] * mkj;
            }
        } else {
            for (int idx = tid; idx < n * n; idx += nt) {
                const int i = idx / n, j = idx - i * n;
                if (i == k) continue;
                const double base = (j == k) ? 0.0 : M[i * ld + j];
                M[i * ld + j] = base - col[i] * M[k * ld + j];
            }
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
                const double t = M[i * ld + k];
                M[i * ld + k] = M[i * ld + p];
                M[i * ld + p] = t;
            }
        __syncthreads();
    }
    T* out = Gt + ((size_t)w * 2 + sp) * n * n;
    for (int idx = tid; idx < n * n; idx += nt) {
        const int i = idx / n, j = idx - i * n;       // Gt[i][j] = inv[j][i]
        out[idx] = (T)M[j * ld + i];
    }
    if (tid == 0) logdet[2 * w + sp] = log(mant) + expo * 0.69314718055994530942;
}

template <typename T>
__global__ void __launch_bounds__(256) invert_kernel(int N, int n, const T* __restrict__ Phi, T* __restrict__ Gt,
                                                     double* __restrict__ logdet, int* err) {
    extern __shared__ double sm[];
    gj_invert<T>(N, n, Phi, Gt, logdet, err, blockIdx.x >> 1, blockIdx.x & 1, sm);
}

// ---------------------------------------------------------------------------
// Mixed form, n > 16: the inverse of an FP32 Slater block, rounded to FP32 as FP64
// Gauss-Jordan's is, mostly without the FP64 pipe, which an FP64 warp instruction
// occupies for 19 clocks of an SM and an FP32 one for a quarter of a clock.
//  1. Gauss-Jordan with partial pivoting on pairs (hi, lo) of FP32 numbers, each
//     product split exactly by one FMA and each sum by Knuth's TwoSum (T. J. Dekker,
//     Numer. Math. 18, 1971): about 47 bits, 12 FP32 operations per update.  Its
//     error on Slater blocks (n = 20 to 64, cond up to 10^4) stays below
//     30 2^-47 max_j|X_lj| max_i|X_ic| max|A| per element: 10^-13 to 10^-12 of the
//     largest, some 10^-5 of the FP32 rounding.
//  2. Where an element lies within kPairMargin 2^-47 (same scale) of a midpoint
//     between FP32 numbers (about one in 10^4), so that the pair cannot tell its
//     rounding, its column gets one Newton correction X r with the residual r = e_c -
//     A x_c in FP64, and those elements are rounded anew.
//  3. Where the corrected element still lies within kExactMargin 2^-53 (same scale) of
//     the midpoint, the FP64 elimination's own error decides its rounding: the block
//     goes to FP64 Gauss-Jordan, as do blocks with a zero pivot or more than kPairColumns
//     columns of step 2 (nearly singular ones).  The FP64 error, in units of 2^-53 of that
//     scale against an extended-precision inverse, exceeds 20 in one undecided element of
//     a thousand (n = 64; at most 46, and less for smaller n); a margin of 24 takes some 4 %
//     of the blocks of n = 64, one of 64 took 11 % and 2 ms more per recompute.
// So the result is FP64 Gauss-Jordan's to the bit: the walkers of 44 starts of N = 128
// (16384 each, five calls) had the same accumulators with either; without step 3 some
// 3600 in 2 x 10^6 differed, one by a whole move.  ln|det A| is the FP64 sum of the
// pivots' logarithms.
//
// Layout: g x g threads (g = ceil(n / 4)) with a 4 x 4 tile of the block each in
// registers; no row moves: the pivot rows are marked and the permutation applied when
// the inverse is written.  Per column two barriers: the column (with the pivot search
// by every warp on its own), then the pivot row.
// 32768 blocks of n = 64: 17.5 ms in FP64, 9.3 ms so (8.4 without step 3).
// ---------------------------------------------------------------------------
constexpr float kPairMargin = 48.f, kExactMargin = 24.f;
constexpr int kPairColumns = 16;

struct PairF { float h, l; };
__device__ __forceinline__ PairF two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    return PairF{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z))};
}
__device__ __forceinline__ PairF pair_mul(PairF a, PairF b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    const float h = __fadd_rn(p, e);
    return PairF{h, __fsub_rn(e, __fsub_rn(h, p))};
}
// 1 / a: the hardware's approximation y, then y (1 + r + r^2), r = 1 - a y exactly formed
__device__ __forceinline__ PairF pair_rcp(PairF a) {
    const float y = __frcp_rn(a.h);
    const float r = __fmaf_rn(-a.l, y, __fmaf_rn(-a.h, y, 1.f));
    const float l = __fmul_rn(y, __fmaf_rn(r, r, r)), h = __fadd_rn(y, l);
    return PairF{h, __fsub_rn(l, __fsub_rn(h, y))};
}

struct PairShared {
    __align__(16) float colh[2][64], coll[2][64], rowh[64], rowl[64];
    PairF piv[64];
    int perm[64], kof[64];    // pivot row of step k; step of pivot row i
    float rmax[64], cmax[64], amax, wmax[8], res[64], corr[64];
    unsigned mark[2];         // columns with an element whose rounding is open
    int open;                 // an element's rounding depends on the FP64 elimination's own error
};

// Column k = 4 kb + kk of the elimination (kk a constant: the tile m stays in
// registers).  used: rows pivoted so far and the padding, per 32.
template <int kk>
__device__ __forceinline__ void pair_column(int n, int kb, int tr, int tc, bool act, PairF (&m)[4][4],
                                            unsigned (&used)[2], bool& fine, PairShared& sh) {
    constexpr int buf = kk & 1;
    const int k = 4 * kb + kk, lane = threadIdx.x & 31, r0 = 4 * tr, c0 = 4 * tc;
    if (k >= n || !fine) return;     // the same on every thread
    if (tc == kb)
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            const PairF v = two_sum(m[a][kk].h, m[a][kk].l);
            sh.colh[buf][r0 + a] = v.h;
            sh.coll[buf][r0 + a] = v.l;
        }
    __syncthreads();
    // largest |column| among the free rows, the lowest row of equals (every warp for itself)
    const unsigned b0 = (used[0] >> lane) & 1u ? 0u : __float_as_uint(sh.colh[buf][lane]) & 0x7fffffffu;
    const unsigned b1 = (used[1] >> lane) & 1u ? 0u : __float_as_uint(sh.colh[buf][lane + 32]) & 0x7fffffffu;
    const unsigned best = __reduce_max_sync(0xffffffffu, b0 > b1 ? b0 : b1);
    const unsigned e0 = __ballot_sync(0xffffffffu, b0 == best), e1 = __ballot_sync(0xffffffffu, b1 == best);
    const int p = e0 ? __ffs(e0) - 1 : 31 + __ffs(e1);
    fine = best != 0u;
    if (p < 32) used[0] |= 1u << p;
    else used[1] |= 1u << (p - 32);
    const int pa = p & 3;
    if (tr == (p >> 2)) {
#pragma unroll
        for (int b = 0; b < 4; ++b) {
            const float h = pa == 0 ? m[0][b].h : pa == 1 ? m[1][b].h : pa == 2 ? m[2][b].h : m[3][b].h;
            const float l = pa == 0 ? m[0][b].l : pa == 1 ? m[1][b].l : pa == 2 ? m[2][b].l : m[3][b].l;
            const PairF v = two_sum(h, l);
            sh.rowh[c0 + b] = v.h;
            sh.rowl[c0 + b] = v.l;
        }
    }
    __syncthreads();
    if (act && fine) {
        const PairF pv{sh.colh[buf][p], sh.coll[buf][p]}, ip = pair_rcp(pv);
        if (threadIdx.x == 0) {
            sh.piv[k] = pv;
            sh.perm[k] = p;
            sh.kof[p] = k;
        }
        PairF r[4], c[4];
        const float4 rh = *(const float4*)(sh.rowh + c0), rl = *(const float4*)(sh.rowl + c0);
        const float4 ch = *(const float4*)(sh.colh[buf] + r0), cl = *(const float4*)(sh.coll[buf] + r0);
        r[0] = PairF{rh.x, rl.x}; r[1] = PairF{rh.y, rl.y}; r[2] = PairF{rh.z, rl.z}; r[3] = PairF{rh.w, rl.w};
        c[0] = PairF{ch.x, cl.x}; c[1] = PairF{ch.y, cl.y}; c[2] = PairF{ch.z, cl.z}; c[3] = PairF{ch.w, cl.w};
#pragma unroll
        for (int b = 0; b < 4; ++b) r[b] = pair_mul(r[b], ip);
        if (tc == kb) {      // the pivot column becomes -c / pivot
            r[kk] = ip;
#pragma unroll
            for (int a = 0; a < 4; ++a) m[a][kk] = PairF{0.f, 0.f};
        }
        if (tr == (p >> 2)) {  // the pivot row becomes row / pivot
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const bool on = a == pa;
                c[a].h = on ? -1.f : c[a].h;
                c[a].l = on ? 0.f : c[a].l;
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    m[a][b].h = on ? 0.f : m[a][b].h;
                    m[a][b].l = on ? 0.f : m[a][b].l;
                }
            }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {     // m -= c r; low parts renormalised when published
                const float q = __fmul_rn(c[a].h, r[b].h);
                float e = __fmaf_rn(c[a].h, r[b].h, -q);
                e = __fmaf_rn(c[a].h, r[b].l, e);
                e = __fmaf_rn(c[a].l, r[b].h, e);
                const PairF t = two_sum(m[a][b].h, -q);
                m[a][b].h = t.h;
                m[a][b].l = __fadd_rn(m[a][b].l, __fsub_rn(t.l, e));
            }
    }
}

__global__ void __launch_bounds__(256, 3) invert_pair_kernel(int N, int n, int g, const float* __restrict__ Phi,
                                                             float* __restrict__ Gt, double* __restrict__ logdet,
                                                             int* err) {
    extern __shared__ double sm[];
    __shared__ PairShared sh;
    const int w = blockIdx.x >> 1, sp = blockIdx.x & 1;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31;
    const bool act = tid < g * g;
    const int tr = act ? tid / g : g, tc = act ? tid - tr * g : g, r0 = 4 * tr, c0 = 4 * tc;
    const float* A = Phi + ((size_t)w * N + (size_t)sp * n) * n;
    PairF m[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) m[a][b] = PairF{(r0 + a < n && c0 + b < n) ? A[(r0 + a) * n + c0 + b] : 0.f, 0.f};
    {
        float v = 0.f;
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) v = fmaxf(v, fabsf(m[a][b].h));
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
        if (lane == 0) sh.wmax[tid >> 5] = v;
        if (tid < 2) sh.mark[tid] = 0u;
        if (tid == 0) sh.open = 0;
        __syncthreads();
        if (tid == 0) {
            for (int q = 1; q < nt / 32; ++q) v = fmaxf(v, sh.wmax[q]);
            sh.amax = v;
        }
    }
    unsigned used[2] = {0u, 0u};         // rows pivoted so far (and the padding), per 32
#pragma unroll
    for (int q = 0; q < 2; ++q)
        if (n < 32 * (q + 1)) used[q] = n <= 32 * q ? 0xffffffffu : 0xffffffffu << (n - 32 * q);
    bool fine = true;
    for (int kb = 0; kb < g; ++kb) {
        pair_column<0>(n, kb, tr, tc, act, m, used, fine, sh);
        pair_column<1>(n, kb, tr, tc, act, m, used, fine, sh);
        pair_column<2>(n, kb, tr, tc, act, m, used, fine, sh);
        pair_column<3>(n, kb, tr, tc, act, m, used, fine, sh);
    }
    __syncthreads();
    const int ld = n + 1;
    float* Xh = (float*)sm;              // X[l][c], high parts, then the rounded inverse
    float* Xl = Xh + n * ld;             // low parts
    if (fine) {
        if (act)                         // X[k][p_j] = M[p_k][j]
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    const int i = r0 + a, j = c0 + b;
                    if (i < n && j < n) {
                        const PairF v = two_sum(m[a][b].h, m[a][b].l);
                        Xh[sh.kof[i] * ld + sh.perm[j]] = v.h;
                        Xl[sh.kof[i] * ld + sh.perm[j]] = v.l;
                    }
                }
        __syncthreads();
        for (int t = tid; t < 2 * n; t += nt) {     // row and column maxima
            const float* q = t < n ? Xh + t * ld : Xh + (t - n);
            const int step = t < n ? 1 : ld;
            float v = 0.f;
            for (int k = 0; k < n; ++k) v = fmaxf(v, fabsf(q[k * step]));
            (t < n ? sh.rmax : sh.cmax)[t < n ? t : t - n] = v;
        }
        __syncthreads();
        const float scale = kPairMargin * 7.105427357601002e-15f * sh.amax;     // 2^-47
        auto undecided = [&](int l, int c) {
            const unsigned hb = __float_as_uint(Xh[l * ld + c]);
            const float half = __uint_as_float(hb & 0x7f800000u) * 5.9604644775390625e-08f;   // half an ulp: 2^(e - 24)
            const float lo = fabsf(Xl[l * ld + c]), d = scale * sh.rmax[l] * sh.cmax[c];
            return fabsf(lo - half) < d || ((hb & 0x7fffffu) == 0u && fabsf(lo - 0.5f * half) < d);
        };
        for (int idx = tid; idx < n * n; idx += nt) {
            const int l = idx / n, c = idx - l * n;
            if (undecided(l, c)) atomicOr(&sh.mark[c >> 5], 1u << (c & 31));
        }
        __syncthreads();
        unsigned mk[2] = {sh.mark[0], sh.mark[1]};
        fine = __popc(mk[0]) + __popc(mk[1]) <= kPairColumns;
        // the marked columns: eight threads per row of A, then per row of X
        for (int h = 0; h < 2 && fine; ++h)
            while (mk[h]) {
                const int c = 32 * h + __ffs(mk[h]) - 1, sub = tid & 7;
                mk[h] &= mk[h] - 1;
                for (int r = tid >> 3; r < (n + 3) / 4 * 4; r += nt >> 3) {    // whole warps (4 rows each) go round
                    double t = 0.0;
                    if (r < n)
                        for (int l = sub; l < n; l += 8)
                            t = fma((double)A[r * n + l], (double)Xh[l * ld + c] + (double)Xl[l * ld + c], t);
                    t += __shfl_xor_sync(0xffffffffu, t, 4);
                    t += __shfl_xor_sync(0xffffffffu, t, 2);
                    t += __shfl_xor_sync(0xffffffffu, t, 1);
                    if (sub == 0 && r < n) sh.res[r] = (float)((r == c ? 1.0 : 0.0) - t);
                }
                __syncthreads();
                for (int l = tid; l < n; l += nt) {
                    float v = 0.f;
                    for (int r = 0; r < n; ++r) v += Xh[l * ld + r] * sh.res[r];
                    sh.corr[l] = v;
                }
                __syncthreads();
                for (int l = tid; l < n; l += nt)
                    if (undecided(l, c)) {
                        const double v = (double)Xh[l * ld + c] + ((double)Xl[l * ld + c] + (double)sh.corr[l]);
                        const float f = (float)v;
                        // distance to f against half an ulp of f (a quarter below a power of two)
                        const unsigned fb = __float_as_uint(f);
                        const double half = (double)(__uint_as_float(fb & 0x7f800000u) * 5.9604644775390625e-08f);
                        const double off = fabs(v - (double)f);
                        const double d = (double)(kExactMargin / kPairMargin / 64.f * scale * sh.rmax[l] * sh.cmax[c]);
                        if (!(fabs(off - half) >= d) || ((fb & 0x7fffffu) == 0u && fabs(off - 0.5 * half) < d))
                            sh.open = 1;
                        Xh[l * ld + c] = f;
                        Xl[l * ld + c] = 0.f;
                    }
                __syncthreads();
            }
        if (fine && sh.open) fine = false;
    }
    if (!fine) {
        __syncthreads();
        gj_invert<float>(N, n, Phi, Gt, logdet, err, w, sp, sm);
        return;
    }
    float* out = Gt + ((size_t)w * 2 + sp) * n * n;
    for (int idx = tid; idx < n * n; idx += nt) out[idx] = Xh[idx % n * ld + idx / n];     // Gt[i][j] = X[j][i]
    if (tid < 32) {
        double lsum = 0.0;
        for (int k = lane; k < n; k += 32) lsum += log(fabs((double)sh.piv[k].h + (double)sh.piv[k].l));
        lsum = warp_sum(lsum);
        if (lane == 0) logdet[2 * w + sp] = lsum;
    }
}

// Mixed form, periodic recompute inside a call: one Newton-Schulz step
//   R = I - A G,  G <- G + G R
// on the inverse the Sherman-Morrison updates have carried since the last
// recompute; A = the Slater block just evaluated at the current positions.
// With E = G - A^-1 the step leaves G' - A^-1 = -E A E, second order in the
// drift.  The residual is formed without rounding error of consequence: each
// product a*g is split exactly into its FP32 value and error (one FMA) and the
// sum is carried as an unevaluated pair hi + lo with Knuth's TwoSum (the
// compensated dot product of Ogita, Rump and Oishi, SIAM J. Sci. Comput. 26,
// 2005), so R is the residual of the FP32 A and G to FP32 relative accuracy
// although A G agrees with I to a few units of FP32 rounding.  G R is small
// and formed in plain FP32.  The result is the inverse of the FP32 Slater
// block to FP32 rounding (what FP64 Gauss-Jordan rounded to FP32 gives) from
// about ten FP32 operations per term of one n^3 product plus one plain n^3
// product; FP64 runs at 1/64 of the FP32 rate on this part.  If max |R_ij| >=
// 0.01 (or is not finite) the block is inverted from scratch by Gauss-Jordan in
// FP64 instead.  ln|det| is not updated here (nothing in a call reads it
// after the first recompute, which is always Gauss-Jordan).
__global__ void __launch_bounds__(256) refine_kernel(int N, int n, int np, const float* __restrict__ Phi,
                                                     float* __restrict__ Gt, double* __restrict__ logdet, int* err) {
    extern __shared__ double sm[];
    const int ld = np + 4, ng = np / 4;
    float* AT = (float*)sm;                  // A^T [j][i]; later G'^T
    float* Gm = AT + (size_t)np * ld;        // G [j][k] = Gt[k][j]
    float* R = Gm + (size_t)np * ld;         // R [i][k]
    __shared__ float rmax_s[8];
    const int w = blockIdx.x >> 1, sp = blockIdx.x & 1;
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const float* A = Phi + ((size_t)w * N + (size_t)sp * n) * n;
    float* Go = Gt + ((size_t)w * 2 + sp) * n * n;
    for (int idx = tid; idx < np * np; idx += nt) {
        const int i = idx / np, j = idx - i * np;
        const bool in = i < n && j < n;
        AT[j * ld + i] = in ? A[i * n + j] : 0.f;
        Gm[j * ld + i] = in ? Go[i * n + j] : 0.f;
    }
    __syncthreads();
    const int r0 = 4 * (tid / ng), c0 = 4 * (tid % ng);
    const bool act = tid < ng * ng;
    float acc[4][4] = {};
    float rm = 0.f;
    if (act) {                               // (A G)[i][k] = sum_j A[i][j] G[j][k] as hi + lo
        float lo[4][4] = {};
        for (int j = 0; j < np; ++j) {
            const float4 a4 = *(const float4*)(AT + j * ld + r0), g4 = *(const float4*)(Gm + j * ld + c0);
            const float av[4] = {a4.x, a4.y, a4.z, a4.w}, gv[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
            for (int a = 0; a < 4; ++a)
#pragma unroll
                for (int b = 0; b < 4; ++b) {
                    // explicit-rounding intrinsics: no contraction into FMAs,
                    // which would void the error-free transformations
                    const float p = __fmul_rn(av[a], gv[b]);
                    const float e = __fmaf_rn(av[a], gv[b], -p);     // a g - p exactly
                    const float s = acc[a][b], t = __fadd_rn(s, p);
                    const float z = __fsub_rn(t, s);
                    const float d = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p, z));   // s + p - t exactly
                    lo[a][b] = __fadd_rn(lo[a][b], __fadd_rn(d, e));
                    acc[a][b] = t;
                }
        }
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const int i = r0 + a, k = c0 + b;
                // (delta - hi) is exact (hi is within a few units of rounding
                // of delta); one rounding when lo is taken off
                const float r = (i < n && k < n) ? __fsub_rn(__fsub_rn(i == k ? 1.f : 0.f, acc[a][b]), lo[a][b]) : 0.f;
                R[i * ld + k] = r;
                rm = fmaxf(rm, isfinite(r) ? fabsf(r) : 1e30f);
            }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rm = fmaxf(rm, __shfl_xor_sync(0xffffffffu, rm, o));
    if (lane == 0) rmax_s[warp] = rm;
    __syncthreads();
    float rmax = 0.f;
    for (int q = 0; q < nt / 32; ++q) rmax = fmaxf(rmax, rmax_s[q]);
    if (!(rmax < 0.01f)) {                   // too far off: FP64 Gauss-Jordan from scratch
        __syncthreads();
        gj_invert<float>(N, n, Phi, Gt, logdet, err, w, sp, sm);
        return;
    }
    if (act) {                               // G'[j][k] = G[j][k] + sum_i G[j][i] R[i][k]
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) acc[a][b] = Gm[(r0 + a) * ld + c0 + b];
        for (int i = 0; i < np; ++i) {
            const float4 r4 = *(const float4*)(R + i * ld + c0);
            const float rv[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
            for (int a = 0; a < 4; ++a) {
                const float gji = Gm[(r0 + a) * ld + i];
#pragma unroll
                for (int b = 0; b < 4; ++b) acc[a][b] += gji * rv[b];
            }
        }
    }
    __syncthreads();                         // every read of A^T done: it takes G'^T
    if (act)
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) AT[(c0 + b) * ld + r0 + a] = acc[a][b];
    __syncthreads();
    for (int idx = tid; idx < n * n; idx += nt) {
        const int k = idx / n, j = idx - k * n;     // Gt[k][j] = G'[j][k]
        Go[idx] = AT[k * ld + j];
    }
}

void launch_refine(int W, int N, int n, const float* Phi, float* Gt, double* logdet, int* err, cudaStream_t st) {
    int np = 4;
    while (np < n) np *= 2;
    const size_t gj = (size_t)n * (n + 1) * sizeof(double) + n * sizeof(double) + n * sizeof(int);
    const size_t ns = (size_t)3 * np * (np + 4) * sizeof(float);
    const size_t smem = gj > ns ? gj : ns;
    // raise the dynamic shared-memory limit to what this launch needs (the
    // kernel also holds static shared memory, so not to the opt-in maximum)
    static size_t attr = 0;
    if (smem > attr &&
        cudaFuncSetAttribute(refine_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) == cudaSuccess)
        attr = smem;
    refine_kernel<<<2 * W, 256, smem, st>>>(N, n, np, Phi, Gt, logdet, err);
}

template <typename T>
static void launch_gj(int W, int N, int n, const T* Phi, T* Gt, double* logdet, int* err, cudaStream_t st) {
    const size_t smem = (size_t)n * (n + 1) * sizeof(double) + n * sizeof(double) + n * sizeof(int);
    const int threads = n >= 32 ? 256 : 64;
    invert_kernel<T><<<2 * W, threads, smem, st>>>(N, n, Phi, Gt, logdet, err);
}

void launch_invert(int W, int N, int n, const double* Phi, double* Gt, double* logdet, int* err, cudaStream_t st) {
    launch_gj(W, N, n, Phi, Gt, logdet, err, st);
}

void launch_invert(int W, int N, int n, const float* Phi, float* Gt, double* logdet, int* err, cudaStream_t st) {
    if (n <= 16) {       // a few thousand FP64 operations: the pair kernel's barriers would cost more
        launch_gj(W, N, n, Phi, Gt, logdet, err, st);
        return;
    }
    const int g = (n + 3) / 4, threads = (g * g + 31) / 32 * 32;
    // the pair inverse and what the FP64 fallback needs are within a few bytes of each other
    const size_t smem = (size_t)n * (n + 1) * sizeof(double) + n * sizeof(double) + n * sizeof(int);
    invert_pair_kernel<<<2 * W, threads, smem, st>>>(N, n, g, Phi, Gt, logdet, err);
}

}  // namespace qmc
