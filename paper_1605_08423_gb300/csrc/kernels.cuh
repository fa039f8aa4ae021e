// kernels.cuh -- host-side launchers of the qmcmd kernels (one per kernel class).
#pragma once
#include "common.cuh"

namespace qmc {

// k_orbitals.cu
void launch_orbitals(const SysView<float>& s, const double* pos, int nrows, float* val, float* grad, float* lap,
                     cudaStream_t st);
// FP64 form, values only; trig: (sin, cos)(pi x / L) [rows][6] of the positions, or null
void launch_orbitals(const SysView<double>& s, const double* pos, const double* trig, int nrows, double* val,
                     cudaStream_t st);
// Thread k of the proposal kernel: electron t (of rows = W N) and what it does there,
// mu = 0..2 a coordinate, 3 the acceptance uniform.  With per_coordinate the 3 rows
// coordinates come first, then the uniforms; else a thread has an electron's all (mu = 3).
// t < 0: nothing to do.  Indices in 64 bits: 4 rows exceeds an int from 2^29 electrons on
// (34 million walkers of N = 16, about 210 GB).
struct ProposeTask { int t, mu; };
__host__ __device__ inline ProposeTask propose_task(long long k, int rows, bool per_coordinate) {
    if (!per_coordinate) return k < rows ? ProposeTask{(int)k, 3} : ProposeTask{-1, 0};
    const long long r3 = 3LL * rows;
    if (k < r3) {
        const long long t = k / 3;
        return ProposeTask{(int)t, (int)(k - 3 * t)};
    }
    return k < r3 + rows ? ProposeTask{(int)(k - r3), 3} : ProposeTask{-1, 0};
}
inline unsigned propose_blocks(int rows, bool per_coordinate, int threads) {
    return (unsigned)(((per_coordinate ? 4LL : 1LL) * rows + threads - 1) / threads);
}
template <typename T>
void launch_propose(int W, int N, double L, double* X, double* Xp, T* ptp, T* uacc, Key key, uint32_t md,
                    uint32_t sweep, double sigma, uint32_t w0, cudaStream_t st);
void launch_init_walkers(int W, int N, double L, const double* R, double* X, Key key, uint32_t w0, cudaStream_t st);

// k_orbitals_tc.cu (tensor-core form of the value-only contraction)
bool tc_orbitals_supported(int n, int B);
void launch_orbitals_tc(const SysView<float>& s, const void* chat, const double* pos, int nrows, float* val,
                        float* grad, float* lap, cudaStream_t st);
void prepare_tc_coeff(const float* C, int B, int n, void* chat, cudaStream_t st);
size_t tc_coeff_bytes(int B, int n);

// k_adjoint_tc.cu (tensor-core form of the orbital part of the force
// estimators; the measure kernel then runs with kt_out/eg_out/elw set)
bool tc_adjoint_supported(int N, int n, int G);
size_t tc_adjoint_coeff_bytes(int n, int G);
void prepare_tc_adjoint_coeff(const float* C, int N, int G, int n, void* ahat, cudaStream_t st);
void launch_adjoint_tc(const SysView<float>& s, const void* ahat, const float* Gt, const float* Kt, const float* eg,
                       const double* elw, const float* frec, double* acc, double* out_dl, double* out_de,
                       cudaStream_t st);

// k_invert.cu: FP64 Gauss-Jordan inverse of each walker's two Slater blocks.
template <typename T>
void launch_invert(int W, int N, int n, const T* Phi, T* Gt, double* logdet, int* err, cudaStream_t st);

// k_invert.cu: mixed-form periodic recompute (one Newton-Schulz step, FP64
// Gauss-Jordan where the carried inverse is too far off).
void launch_refine(int W, int N, int n, const float* Phi, float* Gt, double* logdet, int* err, cudaStream_t st);

// k_sweep.cu: one Metropolis sweep per walker.
// vep: [W][N] per-electron e-n Jastrow sums carried between the sweeps of a
// call (computed when vep_init, i.e. in the call's first sweep).
void launch_sweep(const SysView<float>& s, double* X, const double* Xp, const float* ptp, const float* uacc,
                  const float* Phi, float* Gt, unsigned long long* nacc, float* vep, bool vep_init, cudaStream_t st);
void launch_sweep(const SysView<double>& s, double* X, const double* Xp, const double* ptp, const double* uacc,
                  const double* Phi, double* Gt, unsigned long long* nacc, double* vep, bool vep_init,
                  cudaStream_t st);
// Walkers per CTA for a warp-per-walker kernel that holds at most `most` of them.
int walkers_per_cta(int W, int most);

// k_measure.cu: local energy, d ln psi / dR and dE_L / dR per walker, mixed form.
// ktask [ntask]: structure-factor tasks, (m_x, m_y, first of two |m_z|, index of
// (m_x, m_y, 0)).
// LpY: lap phi rows, overwritten with Y.
// kint [3][nk]: the integer vectors (m_x, m_y, m_z) of the reciprocal vectors.
void launch_measure(const SysView<float>& s, int ntask, const int4* ktask, const float* kint, const double* X,
                    const float* D, float* LpY, const float* Gt, const double* logdet, double* acc, double* out_el, double* out_lnpsi, double* out_dl,
                    double* out_de, float* kt_out, float* eg_out, double* elw, float* rk_out, cudaStream_t st);

// k_measure64.cu: the same in the FP64 form, straight from the inverses (complex
// ones where tv is given: twisted orbitals).  kxyz [3][nk]: the reciprocal vectors.
void launch_measure64(const SysView<double>& s, const TwistView* tv, int ntask, const int4* ktask, const double* kxyz,
                      const double* X, const double* Gt, const double* logdet, double* acc, double* out_el,
                      double* out_lnpsi, double* out_dl, double* out_de, cudaStream_t st);

// k_setup.cu: per-R tables (proton trig, structure factors, p-p Ewald terms; vpp is
// work space [N]) and, with Trec, the reciprocal-space force as a [3N][2 nk]
// matrix on rho(k) (split measure path).
void launch_setup(int N, double L, double kappa, int nk, const int4* kvec, const double* R, double* kw,
                  double* ptrig64, float* ptrig32, double2* eikR, double2* rho_p, double* vconst, double* dvpp,
                  double* vpp, float* R32, float2* eikR32, float* kw32, float* Trec, cudaStream_t st);

// k_setup.cu: real-space Ewald table of the FP64 form (EwTable), once per handle.
void launch_ewald_table(double kappa, double h, double* t, cudaStream_t st);

// k_recforce.cu: F[W][M] = rho[W][K] . T[K][M] (reciprocal-space force of every walker sample).
void launch_recforce_gemm(int W, int M, int K, const float* rho, const float* T, float* F, cudaStream_t st);

// k_reduce.cu: walker reductions and the covariance matrix.
// K walker blocks of W walkers (the twists; else K = 1), each with its own
// result out[K][4 + 3N + 9N^2]; colsum [K][4 + 9N], ws gram_ws_doubles(K, W, N).
void launch_reduce(int K, int W, int N, double moves, const double* acc, const unsigned long long* nacc,
                   double* colsum, double* dev, double* ws, double* out, int* err, cudaStream_t st);
size_t gram_ws_doubles(int K, int W, int N);
// k_reduce.cu: virial pressure of the last call's samples, out [5].
void launch_pressure(int W, int N, const double* acc, const double* vacc, double omega, double T_nuc, double* out,
                     cudaStream_t st);
// k_reduce.cu: walker-sharded form of the same reduction (see there): local
// sums [3 + 9N + 3], then E, f and local deviation sums gram [1 + 9N^2] from
// the summed sums, then E_err and S from the summed gram.
void launch_shard_sums(int W, int N, double moves, const double* acc, const unsigned long long* nacc, double* sums,
                       cudaStream_t st);
void launch_shard_reduce(int W, int N, const double* acc, const double* sums, double* dev, double* ws, double* out,
                         double* gram_out, int* err, cudaStream_t st);
void launch_shard_finish(int N, const double* sums, const double* gram, double* out, cudaStream_t st);

// k_twist.cu: twisted boundary conditions (FP64 form, complex orbitals).
void launch_twist_orbitals(const SysView<double>& s, const TwistView& tv, const double* pos, int nrows, double2* val,
                           cudaStream_t st);
void launch_twist_invert(int W, int N, int n, const double2* Phi, double2* Gt, double* logdet, int* err,
                         cudaStream_t st);
void launch_twist_sweep(const SysView<double>& s, const TwistView& tv, double* X, const double* Xp, const double* ptp,
                        const double* uacc, const double2* Phi, double2* Gt, unsigned long long* nacc, double* vep,
                        bool vep_init, cudaStream_t st);
void launch_twist_average(int K, int N, const double* tout, double* out, cudaStream_t st);
void launch_twist_partial(int Kr, int N, const double* out, double* part, cudaStream_t st);
void launch_twist_combine(int K, int N, const double* part, double* out, cudaStream_t st);

// k_empirical.cu: S = H + mu I, H the Hessian of the screened-Coulomb proton pair potential.
void launch_empirical_s(int N, double L, const double* R, double lambda, double mu, double* S, cudaStream_t st);

// k_langevin.cu (scheme: kLvAdopted, kLvFast or kLvNorogna)
enum : int { kLvAdopted = 0, kLvFast = 1, kLvNorogna = 2 };
void launch_langevin(int n3, double* R, double* Rprev, const double* f, const double* S, double* Sprev,
                     double* Lwork, double T_ha, double delta, double alpha, Key key, uint32_t md, double box,
                     int identity, int scheme, int* err, cudaStream_t st);

// k_langevin.cu: first simplified scheme, predict (y) and correct (R') halves
void launch_first_predict(int n3, const double* R, const double* S, double* Lwork, double T_ha, double delta, Key key,
                          uint32_t md, double* y, int* err, cudaStream_t st);
void launch_first_correct(int n3, double* y, const double* R, const double* f, const double* S, const double* Sy,
                          const double* Lwork, double delta, double box, cudaStream_t st);

// k_toy.cu: rotating-spring toy model, one thread per trajectory (FP64).
struct ToyDev {
    double k, a;          // U = k/2 (|R| - a)^2
    double sr_const;      // radial eigenvalue of S: 1/lambda (G_lambda) or k + mu/lambda (H + mu G_lambda)
    double mu;            // tangential eigenvalue of S is 1 (G_lambda) or k (1 - a/r) + mu
    double T, delta;
    double dt, db;        // adopted scheme: (1 - e^{-alpha D})/alpha, (1 - e^{-2 alpha D})/(2 alpha)
    double half_idb;      // 1 / (2 db)
    double amp, ampb;     // sqrt(2 T D), sqrt(2 T Db)
    int scheme, s_mode, n_steps, n_burn;
    Key key;
};
void launch_toy(const ToyDev& p, int n_traj, const double* xy0, double* out, cudaStream_t st);

}  // namespace qmc
