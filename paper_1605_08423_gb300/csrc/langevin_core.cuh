// langevin_core.cuh -- FP64 building blocks of the accelerated first-order
// Langevin step (SI, integration schemes), shared by the handle's kernels
// (k_langevin.cu) and the allocation-free entry point (k_langevin_static.cu),
// so that all compute the step with the same code.
//
// One thread-block cluster of P CTAs (P = 1 for small n) takes the step.  The
// Cholesky factorisation is blocked: per block column of 32, four warps factor
// the diagonal tile in registers (L D L^T order so that one reciprocal and no
// square root is on the chain), the rows below are solved against it, four warps
// a row tile, and the trailing 32 x 32 tiles are updated by
// all CTAs; the first CTA updates the next diagonal tile first and factors it
// while the others work on the rest.  The matrix stays in L2 (Lc, read and
// written with .cg accesses); the cluster barrier orders the phases.
//
// What bounds it: an SM issues two FP64 multiply-adds a clock, so the n^3/6 of
// n = 384 take 2.3 ms on one SM; 16 SMs bring that under the chain of diagonal
// tiles and barriers.  One CTA, column by column, took 11.5 ms at n = 384 and
// 0.77 ms at n = 48 (0.68 and 0.10 ms in this form).
#pragma once
#include <cooperative_groups.h>

#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

namespace cg = cooperative_groups;

constexpr int kLvThreads = 256, kLvTb = 32;

struct LvSmem {
    double D[kLvTb][kLvTb + 1];   // diagonal tile of the current block column
    double A[kLvTb][kLvTb + 1];   // operand tiles (A also stages a row tile)
    double B[kLvTb][kLvTb + 1];
    double inv[kLvTb];            // reciprocal diagonal of D
    double col[2][kLvTb];         // column being eliminated of a diagonal tile (alternating)
    double yk[2][kLvTb];          // solved block of up to two right-hand sides
    int fail;                     // set by the first CTA: not positive definite
};

// CTAs of the cluster for an n x n factorisation: about as many as the first
// block column has trailing tiles to share.
__host__ inline int langevin_cluster(int n) {
    const int nt = (n + kLvTb - 1) / kLvTb;
    return nt <= 2 ? 1 : nt <= 4 ? 4 : nt <= 7 ? 8 : 16;
}

// Diagonal tile k into sm.D with its reciprocal diagonal (identity beyond n).
__device__ inline void lv_load_diag(int n, const double* Lc, int k, LvSmem& sm) {
    const int k0 = k * kLvTb;
    for (int idx = threadIdx.x; idx < kLvTb * kLvTb; idx += kLvThreads) {
        const int r = idx >> 5, c = idx & 31, i = k0 + r, j = k0 + c;
        const double v = (i < n && j <= i) ? __ldcg(Lc + (size_t)i * n + j) : (r == c ? 1.0 : 0.0);
        sm.D[r][c] = v;
    }
    __syncthreads();
    if (threadIdx.x < kLvTb) sm.inv[threadIdx.x] = 1.0 / sm.D[threadIdx.x][threadIdx.x];
    __syncthreads();
}

// Four warps (threads 0-127): Cholesky factor of diagonal tile k in place.  Lane =
// row, warp q holds columns q, q + 4, ...: the column being eliminated goes through
// shared memory, one named barrier a column, so that the four FP64 issue ports
// share the updates (a lone warp issues one FP64 instruction in 64 clocks; one warp
// for the whole tile took some 50 k clocks).  Returns false on all four warps at a
// pivot that is not positive.
__device__ inline bool lv_factor_tile(int n, double* Lc, int k, LvSmem& sm) {
    constexpr int Q = kLvTb / 4;
    const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5, k0 = k * kLvTb, row = k0 + lane;
    double a[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int c = 4 * q + wq;
        a[q] = (c <= lane && row < n) ? __ldcg(Lc + (size_t)row * n + k0 + c) : (c == lane ? 1.0 : 0.0);
    }
    double dl = 1.0;
    bool ok = true;
#pragma unroll
    for (int c = 0; c < kLvTb; ++c) {
        if (wq == (c & 3)) sm.col[c & 1][lane] = a[c >> 2];
        asm volatile("bar.sync 1, 128;\n" ::: "memory");
        const double* col = sm.col[c & 1];
        const double d = col[c];
        ok = ok && d > 0.0;
        const double y = (d > 1e-280 && d < 1e280) ? qrcp(d) : 1.0 / d;
        if (lane == c) dl = d;
        const double l = col[lane] * y;     // unit-triangular entry; the stored column keeps l d
#pragma unroll
        for (int q = 0; q < Q; ++q) {
            const int j = 4 * q + wq;
            if (j > c) a[q] -= l * col[j];
        }
    }
    if (!ok) return false;
    const double rs = 1.0 / sqrt(dl);
#pragma unroll
    for (int q = 0; q < Q; ++q) {
        const int c = 4 * q + wq;
        const double v = a[q] * __shfl_sync(0xffffffffu, rs, c);
        if (c <= lane && row < n) __stcg(Lc + (size_t)row * n + k0 + c, v);
    }
    return true;
}

// Four warps (wq = 0..3 of them): row tile I of block column k solved against sm.D,
// X = A L_kk^-T; a warp takes 8 rows, its lane 4 r + g row r and columns g, g + 4, ...
__device__ inline void lv_solve_rows(int n, double* Lc, int k, int I, int wq, const LvSmem& sm) {
    constexpr int Q = kLvTb / 4;
    const int lane = threadIdx.x & 31, g = lane & 3, k0 = k * kLvTb, row = I * kLvTb + wq * 8 + (lane >> 2);
    double* p = Lc + (size_t)row * n + k0;
    double b[Q];
#pragma unroll
    for (int q = 0; q < Q; ++q) b[q] = row < n ? __ldcg(p + 4 * q + g) : 0.0;
#pragma unroll
    for (int c = 0; c < kLvTb; ++c) {
        const double x = __shfl_sync(0xffffffffu, b[c >> 2] * sm.inv[c], (lane & 28) | (c & 3));
        if (g == (c & 3)) b[c >> 2] = x;
#pragma unroll
        for (int q = c >> 2; q < Q; ++q)
            if (4 * q + g > c) b[q] -= x * sm.D[4 * q + g][c];
    }
    if (row < n)
#pragma unroll
        for (int q = 0; q < Q; ++q) __stcg(p + 4 * q + g, b[q]);
}

// The CTA: tile (I, J) -= L_Ik L_Jk^T.
__device__ inline void lv_update_tile(int n, double* Lc, int k, int I, int J, LvSmem& sm) {
    const int tid = threadIdx.x, k0 = k * kLvTb, i0 = I * kLvTb, j0 = J * kLvTb;
    __syncthreads();
    for (int idx = tid; idx < kLvTb * kLvTb; idx += kLvThreads) {
        const int r = idx >> 5, c = idx & 31;
        sm.A[r][c] = i0 + r < n ? __ldcg(Lc + (size_t)(i0 + r) * n + k0 + c) : 0.0;
        sm.B[r][c] = j0 + r < n ? __ldcg(Lc + (size_t)(j0 + r) * n + k0 + c) : 0.0;
    }
    const int tx = tid & 15, ty = tid >> 4;
    double v[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
            v[a][b] = (i < n && j <= i) ? __ldcg(Lc + (size_t)i * n + j) : 0.0;
        }
    __syncthreads();
#pragma unroll 8
    for (int c = 0; c < kLvTb; ++c) {
        const double a0 = sm.A[ty][c], a1 = sm.A[ty + 16][c], b0 = sm.B[tx][c], b1 = sm.B[tx + 16][c];
        v[0][0] -= a0 * b0; v[0][1] -= a0 * b1; v[1][0] -= a1 * b0; v[1][1] -= a1 * b1;
    }
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const int i = i0 + ty + 16 * a, j = j0 + tx + 16 * b;
            if (i < n && j <= i) __stcg(Lc + (size_t)i * n + j, v[a][b]);
        }
}

// Block k of the forward solve L y = g (g in shared memory, solved in place), sm.D
// holding diagonal tile k: the block itself by warp 0 (y_k also to sm.yk[0]) ...
__device__ inline void lv_forward_diag(int n, int k, double* g, LvSmem& sm) {
    const int tid = threadIdx.x, k0 = k * kLvTb;
    if (tid < 32) {
        double v = k0 + tid < n ? g[k0 + tid] : 0.0;
#pragma unroll
        for (int c = 0; c < kLvTb; ++c) {
            const double y = __shfl_sync(0xffffffffu, v, c) * sm.inv[c];
            v = tid == c ? y : (tid > c ? v - sm.D[tid][c] * y : v);
        }
        sm.yk[0][tid] = v;
        if (k0 + tid < n) g[k0 + tid] = v;
    }
}
// ... then the rows below, one per thread.
__device__ inline void lv_forward_rows(int n, const double* Lc, int k, double* g, const LvSmem& sm) {
    const int k0 = k * kLvTb;
    for (int i = k0 + kLvTb + threadIdx.x; i < n; i += kLvThreads) {
        const double* p = Lc + (size_t)i * n + k0;
        double s0 = 0, s1 = 0;
#pragma unroll 8
        for (int c = 0; c < kLvTb; c += 2) {
            s0 += __ldcg(p + c) * sm.yk[0][c];
            s1 += __ldcg(p + c + 1) * sm.yk[0][c + 1];
        }
        g[i] -= s0 + s1;
    }
    __syncthreads();
}

// The CTA: back solve L^T x = w for `nrhs` (1 or 2) right-hand sides w[q] in
// shared memory, solved in place.
__device__ inline void lv_backward(int n, const double* Lc, double* const w[2], int nrhs, LvSmem& sm) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int k = (n + kLvTb - 1) / kLvTb - 1; k >= 0; --k) {
        const int k0 = k * kLvTb;
        lv_load_diag(n, Lc, k, sm);
        if (warp < nrhs) {
            double* g = w[warp];
            double v = k0 + lane < n ? g[k0 + lane] : 0.0;
#pragma unroll
            for (int c = kLvTb - 1; c >= 0; --c) {
                const double x = __shfl_sync(0xffffffffu, v, c) * sm.inv[c];
                v = lane == c ? x : (lane < c ? v - sm.D[c][lane] * x : v);
            }
            sm.yk[warp][lane] = v;
            if (k0 + lane < n) g[k0 + lane] = v;
        }
        __syncthreads();
        const int m = n - k0 < kLvTb ? n - k0 : kLvTb;
        for (int j = tid; j < k0; j += kLvThreads) {   // column j of the block's rows: coalesced over threads
            double s0 = 0, s1 = 0;
#pragma unroll 8
            for (int c = 0; c < m; ++c) {
                const double l = __ldcg(Lc + (size_t)(k0 + c) * n + j);
                s0 += l * sm.yk[0][c];
                if (nrhs > 1) s1 += l * sm.yk[1][c];
            }
            w[0][j] -= s0;
            if (nrhs > 1) w[1][j] -= s1;
        }
        __syncthreads();
    }
}

// The cluster: S = L L^T (row-major SPD, lower triangle used) into the lower
// triangle of Lc; where g is set (on the cluster's last CTA only, shared
// memory), the forward solve L y = g runs along, in place.  Returns false on
// every thread if S is not positive definite.
__device__ inline bool lv_cholesky(cg::cluster_group& cl, int n, const double* __restrict__ S, double* Lc, double* g,
                                   LvSmem& sm) {
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int P = (int)cl.num_blocks(), rank = (int)cl.block_rank(), nt = (n + kLvTb - 1) / kLvTb;
    for (int i = rank * (kLvThreads / 32) + warp; i < n; i += P * (kLvThreads / 32))
        for (int j = lane; j <= i; j += 32) __stcg(Lc + (size_t)i * n + j, S[(size_t)i * n + j]);
    if (tid == 0) sm.fail = 0;
    cl.sync();
    if (rank == 0 && warp < 4 && !lv_factor_tile(n, Lc, 0, sm) && tid == 0) sm.fail = 1;
    cl.sync();
    const int* fail = cl.map_shared_rank(&sm.fail, 0);
    for (int k = 0; k < nt; ++k) {
        if (*(volatile const int*)fail) return false;   // written before the last barrier: the same for all
        lv_load_diag(n, Lc, k, sm);
        const int m = nt - 1 - k;                       // row tiles below
        for (int q = rank + P * (warp >> 2); q < m; q += P * (kLvThreads / 128))
            lv_solve_rows(n, Lc, k, k + 1 + q, warp & 3, sm);
        if (g) lv_forward_diag(n, k, g, sm);            // the last CTA has no row tile when P > m
        cl.sync();
        // trailing tiles in column order; the first CTA takes (k+1, k+1) and its
        // factorisation (about a tile's time) and joins once the others have two each
        // (half tiles balance the end better but load as much each: 0.72 ms for 0.68)
        if (rank == 0 && m > 0) {
            lv_update_tile(n, Lc, k, k + 1, k + 1, sm);
            __syncthreads();
            if (warp < 4 && !lv_factor_tile(n, Lc, k + 1, sm) && tid == 0) sm.fail = 1;
        }
        if (g) lv_forward_rows(n, Lc, k, g, sm);
        const int total = m * (m + 1) / 2, head = 2 * (P - 1);
        int J = 0, base = 0;                            // tile t of column J starts at base
        for (int t = 1; t < total; ++t) {
            const int q = t - 1;
            const int owner = P == 1 ? 0 : q < head ? 1 + q % (P - 1) : (q - head) % P;
            if (owner != rank) continue;
            while (t >= base + (m - J)) { base += m - J; ++J; }
            lv_update_tile(n, Lc, k, k + 1 + J + (t - base), k + 1 + J, sm);
        }
        cl.sync();
    }
    return true;
}

// One step of the SI's adopted scheme (or a variant) by one cluster:
//   R' = R + Dt S^{-1} [f - (S_prev - S)(R_prev - R) / (2 Db)] + sqrt(2 T Db) z,  <z z^T> = S^{-1}
// with Dt = (1 - e^{-alpha D})/alpha, Db = (1 - e^{-2 alpha D})/(2 alpha) for
// the adopted scheme with alpha > 0 and Dt = Db = D otherwise; kLvNorogna drops
// the S_prev term; identity != 0 takes S = I (no Cholesky, no S_prev term).
// R_prev - R is the previous step's displacement: in the periodic box (box > 0)
// its minimum image, each component reduced by the nearest multiple of box (a
// position wrapped into the box between the steps would otherwise enter with a
// jump of one box side).
// xi ~ N(0, I) from Philox (counter = (component, md, 0, kLangevin)).
//
// Aliasing: R, Rprev, f, S and Sprev are read and nothing is written to global
// memory except Lc.  R' (r1) and R (r0) are returned in the last CTA's shared
// memory (*owner set there); every CTA's reads of S, Sprev, R, Rprev and f are
// done when the function returns, so the caller may then overwrite them.
// Dynamic shared memory v holds 5 n doubles.  Returns false on every thread if
// S is not positive definite (nothing else is computed then).
__device__ inline bool lv_step(cg::cluster_group& cl, int n, const double* R, const double* Rprev, const double* f,
                               const double* S, const double* Sprev, double* Lc, double T, double delta, double alpha,
                               Key key, uint32_t md, double box, int identity, int scheme, double* v, LvSmem& sm,
                               double** r0_out, double** r1_out) {
    double* g = v;          // [n] drift, then x
    double* dr = g + n;     // [n] R_prev - R
    double* z = dr + n;     // [n] xi, then z
    double* r0 = z + n;     // [n] R
    double* r1 = r0 + n;    // [n] R'
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int P = (int)cl.num_blocks(), rank = (int)cl.block_rank();
    const bool last = rank == P - 1;
    double Dt = delta, Db = delta;
    if (!identity && scheme == kLvAdopted && alpha > 0.0) {
        Dt = (1.0 - exp(-alpha * delta)) / alpha;
        Db = (1.0 - exp(-2.0 * alpha * delta)) / (2.0 * alpha);
    }
    const bool two_time = !identity && scheme != kLvNorogna;
    for (int j = tid; j < n; j += kLvThreads) {
        const double r = R[j];
        r0[j] = r;
        double dj = Rprev[j] - r;
        if (box > 0.0) dj -= box * rint(dj / box);
        dr[j] = dj;
    }
    if (last)
        for (int i = tid; i < n; i += kLvThreads)
            z[i] = Draw<double>::normal(philox((uint32_t)i, md, 0u, kLangevin, key));
    cl.sync();   // every CTA of the cluster runs before its shared memory is written from another
    // g = f - (S_prev - S)(R_prev - R) / (2 Db): a warp per row, into the last CTA's g
    double* gl = cl.map_shared_rank(g, P - 1);
    for (int i = rank * (kLvThreads / 32) + warp; i < n; i += P * (kLvThreads / 32)) {
        double s = 0.0;
        if (two_time) {
            for (int j = lane; j < n; j += 32) s += (Sprev[(size_t)i * n + j] - S[(size_t)i * n + j]) * dr[j];
            s = warp_sum(s);
        }
        if (lane == 0) gl[i] = two_time ? f[i] - s / (2.0 * Db) : f[i];
    }
    if (identity) {
        cl.sync();
    } else {
        if (!lv_cholesky(cl, n, S, Lc, last ? g : nullptr, sm)) {   // its first barrier publishes g
            cl.sync();      // no CTA leaves while another still reads its shared memory
            return false;
        }
        if (last) {
            double* const w[2] = {g, z};
            lv_backward(n, Lc, w, 2, sm);
        }
    }
    if (last) {
        const double amp = T > 0.0 ? sqrt(2.0 * T * Db) : 0.0;
        for (int i = tid; i < n; i += kLvThreads) {
            double r = r0[i] + Dt * g[i] + amp * z[i];
            if (box > 0.0) r -= box * floor(r / box);
            r1[i] = r;
        }
        __syncthreads();
    }
    *r0_out = last ? r0 : nullptr;
    *r1_out = last ? r1 : nullptr;
    return true;
}

// Launch of a cluster kernel with kLvThreads threads per CTA; 16 CTAs need the
// non-portable size, and 8 are taken where the device does not offer it.
template <typename... KArgs, typename... Args>
inline cudaError_t lv_launch(void (*kern)(KArgs...), int P, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kLvThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (P > 8 && cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) {
        cudaGetLastError();
        P = 8;
    }
    static int offers16 = -1;   // whether the device can place the non-portable cluster (same for every kernel here)
    for (;;) {
        at[0].val.clusterDim.x = P;
        at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
        cfg.gridDim = dim3(P);
        int active = 0;
        if (P > 8 && offers16 < 0)
            offers16 = cudaOccupancyMaxActiveClusters(&active, kern, &cfg) == cudaSuccess && active > 0;
        if (P > 8 && !offers16) {
            cudaGetLastError();
            P = 8;
            continue;
        }
        return cudaLaunchKernelEx(&cfg, kern, KArgs(args)...);
    }
}

}  // namespace qmc
