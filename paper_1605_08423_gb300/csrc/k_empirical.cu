// k_empirical.cu -- empirical acceleration matrix S = H + mu I (main text,
// conclusions: S from the Hessian H of an accurate and cheap empirical
// potential, with mu > 0 where H is not positive definite).  H is the Hessian
// of the screened-Coulomb (Yukawa) pair potential of the protons,
//   V = sum_{a<b} sum_{n : |d_ab + nL| < L} v(|d_ab + nL|),  v(r) = exp(-r / lambda) / r,
// images within one box side: the minimum image has |d_mu| <= L/2, so only the
// 8 images with each component either kept or moved by L towards zero can lie
// within L.  Per image vector x, r = |x|:
//   h(x) = v''(r) x x^T / r^2 + v'(r) / r (I - x x^T / r^2),
//   v' = -e (1/r^2 + 1/(lambda r)),  v'' = e (2/r^3 + 2/(lambda r^2) + 1/(lambda^2 r)),  e = exp(-r / lambda);
// block (a, b != a) of H is -sum_images h(x_ab), the diagonal block
// sum_{b != a} sum_images h(x_ab).  FP64.
//
// One block per nucleus a, a thread per partner: the pair's six components go
// to block (a, b), and their sum over the block to block (a, a).  An FP64 exp,
// a square root and divisions per image bound it; a thread per block with the
// whole diagonal sum (N x 27 candidates) on one thread took 2.36 ms at N = 108, this 0.04 ms.
#include "common.cuh"
#include "kernels.cuh"

namespace qmc {

// h[6] = xx, yy, zz, xy, xz, yz of the image sum for the vector d (any image)
__device__ __forceinline__ void yukawa_pair_hessian(double d[3], double L, double il, double h[6]) {
    double sh[3];
#pragma unroll
    for (int mu = 0; mu < 3; ++mu) {
        d[mu] -= L * rint(d[mu] / L);
        sh[mu] = d[mu] >= 0.0 ? -L : L;
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) h[k] = 0.0;
    unsigned mask = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
        const double x = d[0] + ((c & 1) ? sh[0] : 0.0), y = d[1] + ((c & 2) ? sh[1] : 0.0),
                     z = d[2] + ((c & 4) ? sh[2] : 0.0);
        const double r2 = x * x + y * y + z * z;
        if (r2 < L * L && r2 > 0.0) mask |= 1u << c;
    }
    while (mask) {
        const int c = __ffs(mask) - 1;
        mask &= mask - 1;
        const double x = d[0] + ((c & 1) ? sh[0] : 0.0), y = d[1] + ((c & 2) ? sh[1] : 0.0),
                     z = d[2] + ((c & 4) ? sh[2] : 0.0);
        const double r2 = x * x + y * y + z * z;
        const double r = sqrt(r2), ir = 1.0 / r;
        const double e = exp(-r * il);
        const double v1 = -e * (ir * ir + il * ir);
        const double v2 = e * (2.0 * ir * ir * ir + 2.0 * il * ir * ir + il * il * ir);
        const double trans = v1 * ir, radial = (v2 - trans) * ir * ir;
        h[0] += radial * x * x + trans; h[1] += radial * y * y + trans; h[2] += radial * z * z + trans;
        h[3] += radial * x * y; h[4] += radial * x * z; h[5] += radial * y * z;
    }
}

__global__ void __launch_bounds__(128) empirical_s_kernel(int N, double L, const double* __restrict__ R, double lambda,
                                                          double mu, double* __restrict__ S) {
    __shared__ double red[6][32];
    const int a = blockIdx.x, n3 = 3 * N;
    const double il = 1.0 / lambda;
    double acc[6] = {0, 0, 0, 0, 0, 0};
    // packed component of row r, column c
    auto at = [](int r, int c) { return r == c ? r : r + c + 2; };
    for (int b = threadIdx.x; b < N; b += 128) {
        if (b == a) continue;
        double d[3] = {R[3 * a] - R[3 * b], R[3 * a + 1] - R[3 * b + 1], R[3 * a + 2] - R[3 * b + 2]}, h[6];
        yukawa_pair_hessian(d, L, il, h);
#pragma unroll
        for (int k = 0; k < 9; ++k) S[(size_t)(3 * a + k / 3) * n3 + 3 * b + k % 3] = -h[at(k / 3, k % 3)];
#pragma unroll
        for (int k = 0; k < 6; ++k) acc[k] += h[k];
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[k] = block_sum(acc[k], red[k]);
    if (threadIdx.x == 0)
#pragma unroll
        for (int k = 0; k < 9; ++k)
            S[(size_t)(3 * a + k / 3) * n3 + 3 * a + k % 3] = acc[at(k / 3, k % 3)] + (k % 4 == 0 ? mu : 0.0);
}

void launch_empirical_s(int N, double L, const double* R, double lambda, double mu, double* S, cudaStream_t st) {
    empirical_s_kernel<<<N, 128, 0, st>>>(N, L, R, lambda, mu, S);
}

}  // namespace qmc
