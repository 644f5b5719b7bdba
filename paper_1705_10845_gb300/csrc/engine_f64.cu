// Plain-FP64 engine of the recursive Fermi-operator expansion (tanh-doubling
// form) and of its canonical density-matrix perturbation chains.
//
// Products whose result is symmetric (T^2, those of the inverse, 2 T Y, Y M
// for the response) run in symmetric-output mode:
// only upper tiles are computed and mirrored, which halves their cost and
// keeps them exactly symmetric.  Exact symmetry matters: with the A B^T
// product form, an antisymmetric rounding component of Y would be doubled by
// every correction.
//
// The matrices have a leading dimension np that is a multiple of 128, the products run over the N orbitals
// rounded up to 16 only: FP64 multiply-adds are what bounds this engine, and padding to np made 2.1 times
// as many at 400 orbitals and 2.4 times at 96.  Off-diagonal padding is zero, so no sum changes.
#include <cstdio>

#include "precision.h"

namespace xl {
namespace {

#define RET(x)                            \
  do {                                    \
    cudaError_t e_ = (x);                 \
    if (e_ != cudaSuccess) return e_;     \
  } while (0)

class EngineF64 : public Engine {
 public:
  // the block of a matrix that is computed
  struct Dim {
    int n;    // N rounded up to 16
    int ld;   // np
    Dim(int N, const MatSet& m) : n((N + 15) / 16 * 16), ld(m.np) {}
  };

  cudaError_t gemm(cudaStream_t s, Dim d, const double* A, const double* B, double* C, const EpiF64& e, bool sym,
                   double* stats) {
    if (stats) stats[3] += sym ? 0.5 : 1.0;
    RET(prof_begin(s));
    RET(gemm_f64_nt(s, d.n, d.n, d.n, A, d.ld, B, d.ld, C, d.ld, e, sym));
    return prof_end(s, 2.0 * (double)d.n * d.n * d.n * (sym ? 0.5 : 1.0));
  }

  cudaError_t foe(cudaStream_t s, MatSet& m, const double* H, int N, double mu, double sc,
                  const std::vector<LevelPlan>& plan, double* stats, const double*) override {
    const Dim d(N, m);
    const int n = m.n;
    RET(launch_t0_init(s, N, d.n, d.ld, H, mu, sc, m.T[0]));
    // S_k and S_{k-1} alternate between S and T1b, which like A1, Mt and G belongs to the chains and
    // is free here
    double *S = m.S, *Sprev = m.T1b;
    for (int k = 0; k < n; ++k, std::swap(S, Sprev)) {
      const LevelPlan& p = plan[k];
      EpiF64 e1;
      RET(gemm(s, d, m.T[k], m.T[k], S, e1, true, stats));                // S = T^2
      // Y = I - W0 with W_{k-1} = I - Y_{k-1}
      const double* Yp = k > 0 ? m.Y[k - 1] : nullptr;
      RET(launch_combine(s, d.n, d.ld, 1.0 - p.g[0] - p.g[1], p.g[1], Yp, -p.g[2], S, -p.g[3], p.nb > 3 ? Sprev : nullptr,
                         m.Y[k]));
      for (int r = 0; r < p.inv.n; ++r) {
        RET(correct(s, d, m.Y[k], S, -1.0, m.Q, m.A1, m.Mt, m.G, m.Yw, p.inv.order[r], stats));
        std::swap(m.Y[k], m.Yw);
        if (stats) stats[1] += 1;
      }
      EpiF64 et;
      et.alpha = 2.0;
      RET(gemm(s, d, m.T[k], m.Y[k], m.T[k + 1], et, true, stats));       // T_{k+1} = 2 T Y
    }
    return cudaSuccess;
  }

  // One residual correction of Y ~ (I - sg S)^-1 into Yn: R = I - Y + sg Y S, Yn = Y + (R + .. + R^(order-1)) Y.
  // Every factor is a function of one matrix, so each product runs in symmetric-output mode.
  cudaError_t correct(cudaStream_t s, Dim d, const double* Y, const double* S, double sg, double* R, double* R2,
                      double* V, double* U, double* Yn, int order, double* stats) {
    EpiF64 er;
    er.alpha = sg;
    er.E = Y;
    er.lde = d.ld;
    er.beta = -1.0;
    er.diag = 1.0;
    RET(gemm(s, d, Y, S, R, er, true, stats));
    const double* P = R;
    if (order >= 3) {
      EpiF64 e2;
      if (order == 3) {                                                    // P = R + R^2
        e2.E = R;
        e2.lde = d.ld;
        e2.beta = 1.0;
      }
      RET(gemm(s, d, R, R, R2, e2, true, stats));
      P = R2;
    }
    if (order == 5) {                                                      // P = V + V R^2, V = R + R^2
      RET(launch_combine(s, d.n, d.ld, 0.0, 1.0, R, 1.0, R2, 0.0, nullptr, V));
      EpiF64 e5;
      e5.E = V;
      e5.lde = d.ld;
      e5.beta = 1.0;
      RET(gemm(s, d, V, R2, U, e5, true, stats));
      P = U;
    }
    EpiF64 ey;
    ey.E = Y;
    ey.lde = d.ld;
    ey.beta = 1.0;
    return gemm(s, d, P, Y, Yn, ey, true, stats);
  }

  cudaError_t mu_derivative(cudaStream_t s, MuJob& j, double amp) override {
    MatSet& m = *j.m;
    const Dim d(j.N, m);
    const int n = m.n;
    // work matrices of the chains and of the expansion, both idle here
    EpiF64 e1;
    RET(gemm(s, d, m.T[0], m.T[0], m.S, e1, true, j.stats));
    double *Z = m.Yw, *Zn = m.T1b;
    RET(launch_combine(s, d.n, d.ld, j.plan->z0, j.plan->z1, m.S, 0.0, nullptr, 0.0, nullptr, Z));
    for (int r = 0; r < j.plan->inv.n; ++r) {
      RET(correct(s, d, Z, m.S, 1.0, m.Q, m.A1, m.Mt, m.G, Zn, j.plan->inv.order[r], j.stats));
      std::swap(Z, Zn);
    }
    RET(launch_combine(s, d.n, d.ld, -1.0, 2.0, m.Y[n - 1], 0.0, nullptr, 0.0, nullptr, m.Q));   // I - 2 W = 2 Y - I
    RET(gemm(s, d, m.Q, m.Q, m.A1, e1, true, j.stats));
    EpiF64 ea;
    ea.alpha = amp;
    RET(gemm(s, d, m.A1, Z, m.Tmu, ea, true, j.stats));
    return launch_get_diag(s, j.N, d.ld, m.Tmu, j.out_diag);
  }

  cudaError_t chain(cudaStream_t s, MatSet& m, const double* dvec, int N, double* out_diag,
                    double* stats) override {
    const Dim d(N, m);
    const int n = m.n;
    double* T1 = m.T1a;
    double* T1n = m.T1b;
    for (int k = 0; k < n; ++k) {
      const bool last = (k == n - 1);
      EpiF64 em;
      em.alpha = -1.0;
      if (k == 0) {
        RET(launch_level0_A1(s, d.n, d.ld, m.T[0], dvec, m.A1));      // A1 = T0 D + D T0
        em.dvec = dvec;                                         // Mt = 2 D - T_1 A1
        em.ndvec = d.n;
        em.dvec_scale = 2.0;
      } else {
        EpiF64 eg;
        RET(gemm(s, d, m.T[k], T1, m.G, eg, false, stats));   // G = T T1
        RET(launch_transpose_add(s, d.n, d.ld, m.G, m.A1));           // A1 = G + G^T
        em.E = T1;                                              // Mt = 2 T1 - T_{k+1} A1
        em.lde = d.ld;
        em.beta = 2.0;
      }
      RET(gemm(s, d, m.T[k + 1], m.A1, m.Mt, em, false, stats));
      if (last) return launch_row_dot(s, N, d.n, d.ld, m.Y[k], m.Mt, out_diag);   // diag(Y M)
      EpiF64 ey;
      RET(gemm(s, d, m.Y[k], m.Mt, T1n, ey, true, stats));    // T1' = Y M  (= Y Mt^T)
      std::swap(T1, T1n);
    }
    return cudaSuccess;
  }

  cudaError_t trace_tn(cudaStream_t s, MatSet& m, int N, double* out) override {
    return launch_diag_sum(s, N, m.np, m.T[m.n], out);
  }

  cudaError_t density_out(cudaStream_t s, MatSet& m, int N, double dmu, const double*, double* ddiag,
                          double* D) override {
    return launch_density_out_f64(s, N, m.np, m.T[m.n], m.Tmu, dmu, ddiag, D);
  }

  cudaError_t entropy(cudaStream_t s, MatSet& m, int N, double beta, int n_sq, double mu, double dmu,
                      const double* D, const double* H, double* work, double* out) override {
    return launch_entropy_f64(s, m, ent_, N, beta, n_sq, mu, dmu, D, H, work, out);
  }
};

}  // namespace

cudaError_t alloc_matset(MatSet& m, int prec, int np, int n, cudaStream_t s) {
  m.prec = prec;
  m.np = np;
  m.n = n;
  const size_t bytes = sizeof(double) * (size_t)np * np;
  if (prec != 0) return alloc_matset_split(m, s);
  auto A = [&](double** p) -> cudaError_t {
    cudaError_t e = cudaMalloc((void**)p, bytes);
    if (e != cudaSuccess) {
      *p = nullptr;
      return e;
    }
    return cudaMemsetAsync(*p, 0, bytes, s);
  };
  m.T.assign(n + 1, nullptr);
  m.Y.assign(n, nullptr);
  for (auto& p : m.T) RET(A(&p));
  for (auto& p : m.Y) RET(A(&p));
  double** w[] = {&m.S, &m.Q, &m.Yw, &m.G, &m.A1, &m.Mt, &m.T1a, &m.T1b, &m.Tmu};
  for (double** p : w) RET(A(p));
  return cudaSuccess;
}

void free_matset(MatSet& m) {
  for (auto& p : m.T)
    if (p) cudaFree(p);
  for (auto& p : m.Y)
    if (p) cudaFree(p);
  m.T.clear();
  m.Y.clear();
  double** w[] = {&m.S, &m.Q, &m.Yw, &m.G, &m.A1, &m.Mt, &m.T1a, &m.T1b, &m.Tmu};
  for (double** p : w) {
    if (*p) cudaFree(*p);
    *p = nullptr;
  }
  free_matset_split(m);
}

// Default grouped operations: one system after another.
cudaError_t Engine::foe_group(cudaStream_t s, std::vector<FoeJob>& jobs, double sc) {
  for (auto& j : jobs) RET(foe(s, *j.m, j.H, j.N, j.mu, sc, *j.plan, j.stats, j.dpar));
  return cudaSuccess;
}

cudaError_t Engine::mu_derivative_group(cudaStream_t s, std::vector<MuJob>& jobs, double amp) {
  for (auto& j : jobs) RET(mu_derivative(s, j, amp));
  return cudaSuccess;
}

cudaError_t Engine::chain_group(cudaStream_t s, std::vector<ChainJob>& jobs) {
  for (auto& j : jobs) RET(chain(s, *j.m, j.dvec, j.N, j.out_diag, j.stats));
  return cudaSuccess;
}

Engine* make_engine(int prec) {
  if (prec == 0) return new EngineF64();
  return make_split_engine(prec);
}

}  // namespace xl
