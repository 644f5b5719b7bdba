// Internal declarations of the XL-BOMD library (not part of the C ABI).
#pragma once
#include <vector>

#include "common.cuh"

namespace xl {

// Epilogue of C = alpha * A B^T + beta * E + diag * I + diag(dvec):
// E is a matrix with leading dimension lde (may be null), dvec a device
// vector added on the diagonal for i < ndvec (may be null).
struct EpiF64 {
  double alpha = 1.0;
  const double* E = nullptr;
  int lde = 0;
  double beta = 0.0;
  double diag = 0.0;
  const double* dvec = nullptr;
  int ndvec = 0;
  double dvec_scale = 1.0;
};

// FP64 C[M x N] = epi(A[M x K] * B[N x K]^T), row-major, 16-byte aligned rows.  M, N, K multiples
// of 16; the rows of A and B are readable up to the next multiple of 64 (they are loaded for the tiles at
// the edge, and only elements inside M x N are stored).  sym: M == N and only tiles on or above the
// diagonal are computed; each is written to (i, j) and mirrored to (j, i), so
// the result is exactly symmetric (E must then be null or symmetric; it may be C).
// batch > 1: that many products, their matrices a stride apart (st*, elements).
cudaError_t gemm_f64_nt(cudaStream_t s, int M, int N, int K, const double* A, int lda,
                        const double* B, int ldb, double* C, int ldc, const EpiF64& e, bool sym, int batch = 1,
                        size_t stA = 0, size_t stB = 0, size_t stC = 0, size_t stE = 0);

// ---- model (model_kernels.cu) ----
struct ModelConst {
  double eps_s, eps_p, t0[4], r_decay, r_cut, r_taper, U, k;
  double rep_A, rep_rho;   // pair repulsion rep_A exp(-r/rep_rho) S(r); rep_A = 0: off
};

// Positions as pairs of FP32 words (the Coulomb kernels of the split precisions).
cudaError_t launch_split_positions(cudaStream_t s, int nat, const double* R, float2* Rs);
// H0 (np x np, zeroed padding) from positions R (natoms x 3, in [0, L)) in a box L, and a copy of it in H.
cudaError_t launch_build_H0(cudaStream_t s, const ModelConst& m, int nat, double L, const double* R,
                            double* H0, double* H, int np);
// Real-space part of gamma over 27 images of the minimum image (natp x natp, ld natp);
// Rs not null: pair functions in FP32 of 48-bit distances, for the split-precision path.
cudaError_t launch_gamma_real(cudaStream_t s, const ModelConst& m, int nat, double L, double eta,
                              const double* R, const float2* Rs, double* gam, int natp);
// One probe of a response (or one product with gamma): all vectors are of one system.
struct ProbeJob {
  int nat = 0, N = 0, np = 0, natp = 0, kp = 0;
  int unit = -1;                                 // x = e_unit when >= 0 (x and tmp not read)
  const double *gam = nullptr, *SF = nullptr;    // gamma_real and the structure factors (null: no reciprocal part)
  const double* x = nullptr;
  double *tmp = nullptr, *pot = nullptr;         // kp doubles; pot = gamma x
  const double* dmu = nullptr;                   // diagonal of dT_n/dmu
  double *dvec = nullptr, *d1 = nullptr, *w = nullptr;
  double* scal = nullptr;                        // sum d1, sum dmu, mu1; [3] the factor d1 is to be taken back by
  double *Jm = nullptr, *B = nullptr;            // a unit probe's column of J - I and of the identity
};
// Rank-m kernel update (kernel_vec_kernel).  flag may be pinned host memory.
struct KernelVecJob {
  int mode = 0, nat = 0, m = 0;
  double c = 0.0;
  const double* r = nullptr;
  double* V = nullptr;
  const double* W = nullptr;
  double *out = nullptr, *flag = nullptr;
};
// pot = gamma x with gamma = gamma_real + k SF SF^T applied through the structure factors
cudaError_t launch_probe_potential(cudaStream_t s, double k, const std::vector<ProbeJob>& jobs);
// dvec = scale (pot less its average) on orbitals, at a power of two; w (and the column of J - I) from d1
cudaError_t launch_probe_expand(cudaStream_t s, double scale, const std::vector<ProbeJob>& jobs);
cudaError_t launch_probe_finish(cudaStream_t s, const std::vector<ProbeJob>& jobs);
cudaError_t launch_kernel_vec(cudaStream_t s, const std::vector<KernelVecJob>& jobs);
// Structure-factor matrix SF (natp x kp): row I = sqrt(w_g) [cos(G_g.R_I), sin(G_g.R_I)].  Gh: the integer
// vectors h + 8, a byte per component; Gs = sqrt(w_g).
cudaError_t launch_structure_factors(cudaStream_t s, int nat, int ng, double L, const int* Gh, const double* Gs,
                                     const double* R, double* SF, int kp);
// pot[I] = sum_J gamma_IJ x_J  (natoms)
cudaError_t launch_gemv(cudaStream_t s, int nat, const double* gam, int natp, const double* x, double* y);
// H = H0 + diag(pot per orbital); H0 null: H += diag(pot)
cudaError_t launch_apply_potential(cudaStream_t s, int nat, int np, const double* H0, const double* pot,
                                   double* H);
// Gershgorin interval of H: out[0] = min(H_ii - r_i), out[1] = max(H_ii + r_i)
cudaError_t launch_gershgorin(cudaStream_t s, int n, int np, const double* H, double* out);
// Forces: band part from D (np x np), pair repulsion (rep_A != 0), Coulomb real-space and reciprocal parts
// (SF: structure factors of R; work: 2 kp + 3 nat force_parts(nat) doubles).  Rs as for launch_gamma_real.
int force_parts(int nat);
cudaError_t launch_forces(cudaStream_t s, const ModelConst& m, int nat, double L, double eta, int ng,
                          const double* G4, const double* R, const float2* Rs, const double* SF, int kp,
                          const double* D, int np, const double* q, const double* n, double* F, double* work);
// Pair repulsion: e_I = half the pair energy of atom I (E_rep = sum_I e_I).
cudaError_t launch_repulsion_energy(cudaStream_t s, const ModelConst& m, int nat, double L, const double* R,
                                    double* e);
// q_I = sum_{a in I} (1 + Tn_aa) + 2 dmu dmu_diag_a - Z_I, r = q - n
cudaError_t launch_charges(cudaStream_t s, int nat, const double* ddiag, const double* Z,
                           const double* n, double* q, double* r);
// Verlet (Eqs. Integration, VRL_Damp): first half kick + drift + n update.
cudaError_t launch_verlet_first(cudaStream_t s, int nat, double L, double dt, double mass_inv_acc,
                                double* R, double* V, const double* F, double* nh, int kmax,
                                const double* Kr, double kappa, double alpha, const double* c);
cudaError_t launch_verlet_second(cudaStream_t s, int nat, double dt, double mass_inv_acc, double* V,
                                 const double* F);

// ---- expansion helpers (foe_kernels.cu), FP64: over the leading m x m block, leading dimension np ----
cudaError_t launch_t0_init(cudaStream_t s, int n, int m, int np, const double* H, double mu, double scale,
                           double* T0);
cudaError_t launch_level0_A1(cudaStream_t s, int m, int np, const double* T0, const double* d, double* A1);
cudaError_t launch_transpose_add(cudaStream_t s, int m, int np, const double* G, double* A1);
cudaError_t launch_row_dot(cudaStream_t s, int n, int k, int np, const double* Y, const double* M, double* out);
cudaError_t launch_get_diag(cudaStream_t s, int n, int np, const double* X, double* out);
// out[slot] = sum_{i<n} x[i] (deterministic, one block)
cudaError_t launch_sum(cudaStream_t s, int n, const double* x, double* out);
// out = sum_{i,j<n} A_ij B_ij (deterministic two-level reduction; work >= 1024 doubles)
cudaError_t launch_frob_dot(cudaStream_t s, int n, int np, const double* A, const double* B, double* work,
                            double* out);
// Energy parts: out[0..] from vectors (Coulomb, kinetic).
cudaError_t launch_energy_vec(cudaStream_t s, int nat, const double* q, const double* n,
                              const double* pot, const double* V, double mass, double* out);

}  // namespace xl
