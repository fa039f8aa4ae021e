// k_reduce.cu -- walker reductions: E, its error bar, the mean force and the
// covariance matrix S of the paper's covariance definition,
//   f   = -<dE_L/dR> - 2(<E_L dlnpsi/dR> - E <dlnpsi/dR>)
//   f_w = same with the means of walker w (global E)
//   S   = sum_w (f_w - f)(f_w - f)^T / (W (W-1))     (covariance of the mean)
//   E_err^2 = sum_w (E_w - E)^2 / (W (W-1)),  N_c = number of samples.
// FP64, fixed-order trees (bitwise reproducible; no atomics).
// Output layout: [E, E_err, N_c, accept, f(3N), S(3N x 3N)].
//
// Walker-sharded form (walkers split over processes, one GPU each): the same
// reduction in three steps around two sums over the processes --
//   local column sums (plus walkers and moves)          -> summed over processes
//   E, f from the global sums; local sums of (E_w - E)^2 and of
//   (f_w - f)(f_w - f)^T with the global E, f          -> summed over processes
//   E_err and S from the global sums and walker count.
// The result equals the single-process reduction over all walkers up to the
// order of the FP64 sums.
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// The reductions run for a batch of K walker blocks of W walkers each (the
// twists of a twisted handle; K = 1 otherwise): one launch sequence for the whole
// mesh, where one per twist made 320 launches and 2.25 ms of a 64-twist call at N = 64
// (0.29 ms batched).  The batch is part of blockIdx.x, the one grid dimension that goes
// beyond 65535: a 41 x 41 x 41 mesh has 68921 twists.

// colsum[c] = sum_w acc[w][c] for c < ncol; colsum[ncol] = sum_w nacc[w].
__global__ void colsum_kernel(int W, int ncol, const double* __restrict__ acc, const unsigned long long* __restrict__ nacc,
                              double* colsum) {
    __shared__ double red[32];
    const int c = blockIdx.x % (ncol + 1), b = blockIdx.x / (ncol + 1);
    acc += (size_t)b * W * ncol;
    nacc += (size_t)b * W;
    colsum += (size_t)b * (ncol + 1);
    double s = 0.0;
    if (c < ncol)
        for (int w = threadIdx.x; w < W; w += blockDim.x) s += acc[(size_t)w * ncol + c];
    else
        for (int w = threadIdx.x; w < W; w += blockDim.x) s += (double)nacc[w];
    s = block_sum(s, red);
    if (threadIdx.x == 0) colsum[c] = s;
}

// E, f, N_c and the acceptance ratio from column sums (moves < 0: read the
// number of moves from colsum[ncol + 2], as the sharded form stores it).
__global__ void finalize_kernel(int N, double moves, const double* __restrict__ colsum, double* out, int* err) {
    const int N3 = 3 * N, ncol = 3 + 9 * N;
    colsum += (size_t)blockIdx.x * (ncol + 1);
    out += (size_t)blockIdx.x * (4 + N3 + (size_t)N3 * N3);
    const double cnt = colsum[0];
    const double E = colsum[1] / cnt;
    for (int c = threadIdx.x; c < N3; c += blockDim.x) {
        const double f = -colsum[3 + 2 * N3 + c] / cnt - 2.0 * (colsum[3 + N3 + c] / cnt - E * colsum[3 + c] / cnt);
        out[4 + c] = f;
        if (!isfinite(f)) raise_err(err, kErrNonfinite);
    }
    if (threadIdx.x == 0) {
        out[0] = E;
        out[2] = cnt;
        out[3] = colsum[ncol] / (moves < 0.0 ? colsum[ncol + 2] : moves);
        if (!isfinite(E)) raise_err(err, kErrNonfinite);
    }
}

// dev[w][c] = f_w[c] - f[c] (c < 3N), dev[w][3N] = E_w - E.
__global__ void deviation_kernel(int W, int N, int blocks, const double* __restrict__ acc, const double* __restrict__ out,
                                 double* dev) {
    const int N3 = 3 * N, ncol = 3 + 9 * N;
    const int b = blockIdx.x / blocks;                     // `blocks` blocks a batch
    const size_t t = (size_t)(blockIdx.x - b * blocks) * blockDim.x + threadIdx.x;
    if (t >= (size_t)W * (N3 + 1)) return;
    acc += (size_t)b * W * ncol;
    out += (size_t)b * (4 + N3 + (size_t)N3 * N3);
    dev += (size_t)b * W * (N3 + 1);
    const int w = (int)(t / (N3 + 1)), c = (int)(t - (size_t)w * (N3 + 1));
    const double* a = acc + (size_t)w * ncol;
    const double cnt = a[0], E = out[0];
    if (c < N3) {
        const double fw = -a[3 + 2 * N3 + c] / cnt - 2.0 * (a[3 + N3 + c] / cnt - E * a[3 + c] / cnt);
        dev[t] = fw - out[4 + c];
    } else {
        dev[t] = a[1] / cnt - E;
    }
}

// Gram matrix of the deviations, sum_w dev[w][i] dev[w][j], and sum_w (E_w -
// E)^2.  The FP64 pipe bounds it (3N (3N + 1) / 2 multiply-adds a walker): only
// the lower triangle is formed, in 16 x 16 tiles of one output a thread, and
// the walkers of a tile are cut into nsplit slices so that the chip is filled
// at every N (32 x 32 tiles of the whole matrix left 144 blocks at N = 128 and
// 36 at N = 64: the reduction took 5.5 ms for 16384 walkers and 1.3 ms for 4096,
// now 2.5 and 0.24 ms).  The slices'
// partial tiles go to ws [K][nsplit][tiles][256], summed in order by
// gram_sum_kernel.  blockIdx.x counts tiles (the last one is the energy's sum),
// then slices, then batches.
constexpr int kGramTile = 16, kGramRows = 32;
__global__ void __launch_bounds__(256) gram_kernel(int W, int N, int tiles, int ns, const double* __restrict__ dev, double* ws) {
    __shared__ double A[kGramRows][kGramTile], Bm[kGramRows][kGramTile];
    const int N3 = 3 * N, ld = N3 + 1, tid = threadIdx.x;
    const int q = blockIdx.x / (tiles + 1), t = blockIdx.x - q * (tiles + 1), b = q / ns, sl = q - b * ns;
    dev += (size_t)b * W * ld;
    ws += (size_t)blockIdx.x * 256;
    const int w0 = (int)((long long)W * sl / ns), w1 = (int)((long long)W * (sl + 1) / ns);
    if (t == tiles) {
        double e = 0.0;
        for (int w = w0 + tid; w < w1; w += 256) {
            const double d = dev[(size_t)w * ld + N3];
            e += d * d;
        }
        ws[tid] = e;
        return;
    }
    int I = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= t) ++I;
    while (I * (I + 1) / 2 > t) --I;
    const int i0 = kGramTile * I, j0 = kGramTile * (t - I * (I + 1) / 2);
    const int tx = tid & 15, ty = tid >> 4;
    double s0 = 0.0, s1 = 0.0;
    for (int wb = w0; wb < w1; wb += kGramRows) {
#pragma unroll
        for (int r = ty; r < kGramRows; r += 16) {
            const int w = wb + r;
            A[r][tx] = (w < w1 && i0 + tx < N3) ? dev[(size_t)w * ld + i0 + tx] : 0.0;
            Bm[r][tx] = (w < w1 && j0 + tx < N3) ? dev[(size_t)w * ld + j0 + tx] : 0.0;
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < kGramRows; r += 2) {
            s0 += A[r][ty] * Bm[r][tx];
            s1 += A[r + 1][ty] * Bm[r + 1][tx];
        }
        __syncthreads();
    }
    ws[tid] = s0 + s1;
}

// dst_S[i][j] = dst_S[j][i] = scale * (sum of the tile's slices); *dst_e gets
// sqrt(scale * sum_w (E_w - E)^2) when finish != 0, else the plain sum.  Per
// batch dst_S and dst_e advance by `stride`.
__global__ void __launch_bounds__(256) gram_sum_kernel(int N, int tiles, int ns, const double* __restrict__ ws,
                                                       double* dst_e, double* dst_S, size_t stride, double scale,
                                                       int finish) {
    __shared__ double red[32];
    const int N3 = 3 * N, tid = threadIdx.x, b = blockIdx.x / (tiles + 1), t = blockIdx.x - b * (tiles + 1);
    dst_e += b * stride;
    dst_S += b * stride;
    ws += ((size_t)b * ns * (tiles + 1) + t) * 256 + tid;
    double v = 0.0;
    for (int s = 0; s < ns; ++s) v += ws[(size_t)s * (tiles + 1) * 256];
    if (t == tiles) {
        v = block_sum(v, red);
        if (tid == 0) *dst_e = finish ? sqrt(v * scale) : v;
        return;
    }
    int I = (int)((sqrtf(8.f * t + 1.f) - 1.f) * 0.5f);
    while ((I + 1) * (I + 2) / 2 <= t) ++I;
    while (I * (I + 1) / 2 > t) --I;
    const int i = kGramTile * I + (tid >> 4), j = kGramTile * (t - I * (I + 1) / 2) + (tid & 15);
    if (i >= N3 || j >= N3) return;
    v *= scale;
    dst_S[(size_t)i * N3 + j] = v;
    dst_S[(size_t)j * N3 + i] = v;
}

static int gram_tiles(int N) {
    const int nt = (3 * N + kGramTile - 1) / kGramTile;
    return nt * (nt + 1) / 2;
}
// Slices per tile: about six blocks an SM of 152 in all, at least 64 walkers each.
static int gram_splits(int K, int W, int N) {
    const int want = (912 + gram_tiles(N) * K - 1) / (gram_tiles(N) * K), most = W / 64;
    return want < 1 || most < 1 ? 1 : (want < most ? want : most);
}
size_t gram_ws_doubles(int K, int W, int N) {
    return (size_t)K * gram_splits(K, W, N) * (gram_tiles(N) + 1) * 256;
}

static void gram(int K, int W, int N, const double* dev, double* ws, double* dst_e, double* dst_S, size_t stride,
                 double scale, int finish, cudaStream_t st) {
    const int tiles = gram_tiles(N), ns = gram_splits(K, W, N);
    gram_kernel<<<(unsigned)(tiles + 1) * ns * K, 256, 0, st>>>(W, N, tiles, ns, dev, ws);
    gram_sum_kernel<<<(unsigned)(tiles + 1) * K, 256, 0, st>>>(N, tiles, ns, ws, dst_e, dst_S, stride, scale, finish);
}

static void deviations(int K, int W, int N, const double* acc, const double* out, double* dev, cudaStream_t st) {
    const size_t tot = (size_t)W * (3 * N + 1);
    const int blocks = (int)((tot + 255) / 256);
    deviation_kernel<<<(unsigned)blocks * K, 256, 0, st>>>(W, N, blocks, acc, out, dev);
}

void launch_reduce(int K, int W, int N, double moves, const double* acc, const unsigned long long* nacc, double* colsum,
                   double* dev, double* ws, double* out, int* err, cudaStream_t st) {
    const int ncol = 3 + 9 * N, N3 = 3 * N;
    colsum_kernel<<<(unsigned)(ncol + 1) * K, 256, 0, st>>>(W, ncol, acc, nacc, colsum);
    finalize_kernel<<<K, 256, 0, st>>>(N, moves, colsum, out, err);
    deviations(K, W, N, acc, out, dev, st);
    gram(K, W, N, dev, ws, out + 1, out + 4 + N3, 4 + N3 + (size_t)N3 * N3, W > 1 ? 1.0 / ((double)W * (W - 1)) : 0.0, 1,
         st);
}

// ---------------------------------------------------------------------------
// Walker-sharded form.
// ---------------------------------------------------------------------------
__global__ void shard_counts_kernel(int N, double walkers, double moves, double* sums) {
    const int ncol = 3 + 9 * N;
    sums[ncol + 1] = walkers;
    sums[ncol + 2] = moves;
}

// E_err and S from the summed partial sums: scale by 1 / (W (W - 1)), W the
// summed walker count.
__global__ void shard_finish_kernel(int N, const double* __restrict__ sums, const double* __restrict__ gram,
                                    double* out) {
    const int N3 = 3 * N, ncol = 3 + 9 * N;
    const double W = sums[ncol + 1];
    const double scale = W > 1.0 ? 1.0 / (W * (W - 1.0)) : 0.0;
    const size_t tot = (size_t)N3 * N3;
    for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < tot; i += (size_t)gridDim.x * blockDim.x)
        out[4 + N3 + i] = gram[1 + i] * scale;
    if (blockIdx.x == 0 && threadIdx.x == 0) out[1] = sqrt(gram[0] * scale);
}

// Virial pressure of the last call's samples (the potential is homogeneous of
// degree -1 in all lengths -- the Ewald sum with kappa L and the k cutoff in
// units of 2 pi / L fixed included -- so for the trial state scaled with the
// box, E(lambda) = T / lambda^2 + V / lambda and -dE/dOmega = (2 T + V) / (3 Omega)):
//   P_w = (2 E_w - V_w) / (3 Omega)   per walker (T = E - V),
//   P   = (2 E - V) / (3 Omega) + N T_nuc / Omega   (classical nuclei, ideal-gas term),
//   P_err^2 = sum_w (P_w - P_el)^2 / (W (W - 1)).
// out = [P, P_err, P_el, <V_L>, <T_L>] (hartree / bohr^3, hartree).
__global__ void pressure_kernel(int W, int N, const double* __restrict__ acc, const double* __restrict__ vacc,
                                double omega, double T_nuc, double* out) {
    __shared__ double red[32];
    const int ncol = 3 + 9 * N;
    double c = 0.0, e = 0.0, v = 0.0;
    for (int w = threadIdx.x; w < W; w += blockDim.x) {
        c += acc[(size_t)w * ncol];
        e += acc[(size_t)w * ncol + 1];
        v += vacc[w];
    }
    c = block_sum(c, red);
    e = block_sum(e, red);
    v = block_sum(v, red);
    const double E = e / c, V = v / c;
    const double Pel = (2.0 * E - V) / (3.0 * omega);
    double d2 = 0.0;
    for (int w = threadIdx.x; w < W; w += blockDim.x) {
        const double cw = acc[(size_t)w * ncol];
        const double pw = (2.0 * acc[(size_t)w * ncol + 1] / cw - vacc[w] / cw) / (3.0 * omega);
        d2 += (pw - Pel) * (pw - Pel);
    }
    d2 = block_sum(d2, red);
    if (threadIdx.x == 0) {
        out[0] = Pel + N * T_nuc / omega;
        out[1] = W > 1 ? sqrt(d2 / ((double)W * (W - 1))) : 0.0;
        out[2] = Pel;
        out[3] = V;
        out[4] = E - V;
    }
}

void launch_pressure(int W, int N, const double* acc, const double* vacc, double omega, double T_nuc, double* out,
                     cudaStream_t st) {
    pressure_kernel<<<1, 256, 0, st>>>(W, N, acc, vacc, omega, T_nuc, out);
}

void launch_shard_sums(int W, int N, double moves, const double* acc, const unsigned long long* nacc, double* sums,
                       cudaStream_t st) {
    const int ncol = 3 + 9 * N;
    colsum_kernel<<<ncol + 1, 256, 0, st>>>(W, ncol, acc, nacc, sums);
    shard_counts_kernel<<<1, 1, 0, st>>>(N, (double)W, moves, sums);
}

void launch_shard_reduce(int W, int N, const double* acc, const double* sums, double* dev, double* ws, double* out,
                         double* gram_out, int* err, cudaStream_t st) {
    finalize_kernel<<<1, 256, 0, st>>>(N, -1.0, sums, out, err);
    deviations(1, W, N, acc, out, dev, st);
    gram(1, W, N, dev, ws, gram_out, gram_out + 1, 0, 1.0, 0, st);
}

void launch_shard_finish(int N, const double* sums, const double* gram, double* out, cudaStream_t st) {
    shard_finish_kernel<<<64, 256, 0, st>>>(N, sums, gram, out);
}

}  // namespace qmc
