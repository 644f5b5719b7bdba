// Electronic entropy of the occupations of D without eigenvalues (energy
// monitor, Eq. S_entropy).
//
// With f = (1 + t_n)/2 and the tanh-doubling map, ln(f/(1-f)) = 2^(n+1)
// artanh(t_0), and 1 - f satisfies ln(1 - x_{k+1}) = 2 ln(1 - x_k) - ln b_k
// with b_k = (1 + t_k^2)/2.  Summed over eigenstates:
//   sum_i s(f_i) = -sum ln(1 - f_i) - Tr[D 2^(n+1) artanh(T_0)]
//   sum ln(1 - f_i) = 2^n logdet(I - T_0) + sum_k 2^(n-1-k) logdet(Y_k) - N ln 2
// where Y_k = (I + T_k^2)^-1.  Every logdet is of a well-conditioned SPD
// matrix (spectra in [1 - |t_0|max, 1 + |t_0|max] and [1/2, 1]) and is taken
// by a blocked FP64 Cholesky factorisation; artanh(T_0) is its odd power
// series (|t_0| << 1), whose traces against D come from Frobenius products.
#include <algorithm>
#include <cmath>
#include <functional>

#include "precision.h"

namespace xl {
namespace {

#define RET(x)                        \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

constexpr int CB = EntropyWork::kPanel;

// Diagonal block (kb, kb) of matrix blockIdx.x: A = L D L^T (L unit lower); part[..][kb / CB] = sum ln d (NaN for
// a non-positive pivot) and Li = D^-1/2 L^-1, for which A^-1 = Li^T Li.  In place: at step j column j
// turns from A's into L^-1's, its old values are in col[j & 1].
__global__ void __launch_bounds__(256) chol_panel_kernel(const double* __restrict__ W, size_t stride, int np, int kb,
                                                         double* __restrict__ Li, double* __restrict__ part, int npart) {
  __shared__ double x[CB][CB + 1], col[2][CB], d[CB], inv;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const double* A = W + stride * blockIdx.x;
  for (int e = tid; e < CB * CB; e += 256) x[e / CB][e % CB] = A[(size_t)(kb + e / CB) * np + kb + e % CB];
  __syncthreads();
  if (tid < CB) col[0][tid] = x[tid][0];
  if (tid == 0) {
    d[0] = x[0][0];
    inv = 1.0 / x[0][0];
  }
  __syncthreads();
  for (int j = 0; j < CB - 1; ++j) {
    const double* cj = col[j & 1];
    double* cn = col[(j + 1) & 1];
    const double iv = inv;
    __syncthreads();   // every thread has read inv
    for (int i = j + 1 + ty; i < CB; i += 16) {
      const double l = cj[i] * iv;
      for (int c = tx; c <= i; c += 16) {
        if (c == j) {
          x[i][j] = -l;
          continue;
        }
        const double v = x[i][c] - l * (c < j ? x[j][c] : cj[c]);
        x[i][c] = v;
        if (c == j + 1) {
          cn[i] = v;
          if (i == j + 1) {
            d[i] = v;
            inv = 1.0 / v;
          }
        }
      }
    }
    __syncthreads();
  }
  if (tid < CB) {
    const double v = d[tid];
    const double s = warp_sum(v > 0.0 ? log(v) : nan(""));
    if ((tid & 31) == 0) col[0][tid >> 5] = s;
    col[1][tid] = 1.0 / sqrt(v);
  }
  __syncthreads();
  if (tid == 0) part[(size_t)npart * blockIdx.x + kb / CB] = col[0][0] + col[0][1];
  double* out = Li + (size_t)CB * CB * blockIdx.x;
  for (int e = tid; e < CB * CB; e += 256) {
    const int i = e / CB, c = e % CB;
    out[e] = c < i ? x[i][c] * col[1][i] : c == i ? col[1][i] : 0.0;
  }
}

// out[b] = sum of the panels' parts of matrix b
__global__ void chol_sum_kernel(int npart, const double* __restrict__ part, double* __restrict__ out) {
  __shared__ double sh[32];
  double v = 0.0;
  for (int i = threadIdx.x; i < npart; i += blockDim.x) v += part[(size_t)npart * blockIdx.x + i];
  v = block_sum(v, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = v;
}

// Y on the N x N block, the identity around it: log det of the whole is that of the block
__global__ void block_or_identity_kernel(size_t count, int N, int np, const double* __restrict__ Y,
                                         double* __restrict__ dst) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= count) return;
  const int i = (int)(idx / np), j = (int)(idx % np);
  dst[idx] = (i < N && j < N) ? Y[idx] : (i == j ? 1.0 : 0.0);
}

// W = I - T (np x np)
__global__ void ident_minus_f64_kernel(size_t count, int np, const double* __restrict__ T, double* __restrict__ W) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= count) return;
  const int i = (int)(idx / np), j = (int)(idx % np);
  W[idx] = (i == j ? 1.0 : 0.0) - T[idx];
}

struct EntW {
  double w_ld[42];   // weights of the logdet slots
  double w_tr[8];    // weights of the trace slots
  int nld, ntr;
  double cst;        // N ln 2
};

// out = cst - sum_k w_ld[k] ld[k] - sum_j w_tr[j] tr[j]
__global__ void entropy_combine_kernel(EntW w, const double* __restrict__ ld, const double* __restrict__ tr,
                                       double* __restrict__ out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double s = w.cst;
  for (int k = 0; k < w.nld; ++k) s -= w.w_ld[k] * ld[k];
  for (int j = 0; j < w.ntr; ++j) s -= w.w_tr[j] * tr[j];
  *out = s;
}

// log-determinants of the leading m x m blocks (m a multiple of CB) of the nb SPD matrices in the work area
// (destroyed) into out[0..nb)
cudaError_t logdet_spd(cudaStream_t s, const EntropyWork& w, int m, int np, int nb, double* out) {
  const size_t cnt = (size_t)np * np;
  const int npart = m / CB;
  for (int kb = 0; kb < m; kb += CB) {
    chol_panel_kernel<<<nb, 256, 0, s>>>(w.mats, cnt, np, kb, w.li, w.part, npart);
    note_launch();
    RET(cudaGetLastError());
    const int rest = m - kb - CB;
    if (rest > 0) {
      // X = A21 Li^T, A22 -= X X^T
      double* A21 = w.mats + (size_t)(kb + CB) * np + kb;
      EpiF64 ex;
      RET(gemm_f64_nt(s, rest, CB, CB, A21, np, w.li, CB, w.rows, CB, ex, false, nb, cnt, (size_t)CB * CB,
                      (size_t)np * CB));
      EpiF64 e;
      e.alpha = -1.0;
      e.E = A21 + CB;
      e.lde = np;
      e.beta = 1.0;
      RET(gemm_f64_nt(s, rest, rest, CB, w.rows, CB, w.rows, CB, A21 + CB, np, e, true, nb, (size_t)np * CB,
                      (size_t)np * CB, cnt, cnt));
    }
  }
  chol_sum_kernel<<<nb, 128, 0, s>>>(npart, w.part, out);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

// Entropy from FP64 inputs.  T0: FP64 T_0; load_Y(k, dst) writes Y_k as an
// FP64 matrix into dst; S, Q, Yw, A1, Mt: FP64 work matrices (np x np);
// nterms: terms j = 0..nterms-1 of the artanh series.
cudaError_t entropy_fp64(cudaStream_t s, int N, int np, int n, int n_sq, const double* T0,
                         const std::function<cudaError_t(int, double*)>& load_Y, EntropyWork& area, double* S, double* Q,
                         double* Yw, double* A1, double* Mt, int nterms, const double* D, double* work,
                         double* out) {
  if (n + 1 > 42 || nterms < 1 || nterms > 6) return cudaErrorInvalidValue;
  // work layout: [0, 64): logdet slots, [64, 72): trace slots, [1024, 2048): Frobenius partials
  double* ld = work;
  double* tr = work + 64;
  double* fwork = work + 1024;
  const size_t count = (size_t)np * np;
  const int mc = (N + CB - 1) / CB * CB, m = (N + 15) / 16 * 16;   // padding does not change what follows
  // logdet(I - T_0), then logdet(Y_k)
  area.reserve(np, n + 1,
               [](size_t bytes) -> void* {
                 void* p = nullptr;
                 if (cudaMalloc(&p, bytes) == cudaSuccess) return p;
                 cudaGetLastError();   // a smaller area is asked for next
                 return nullptr;
               },
               [](void* p) { cudaFree(p); });
  const EntropyWork ew = area.cap > 0 ? area : EntropyWork::on(S, Q, np);
  for (int k0 = 0; k0 <= n; k0 += ew.cap) {
    const int nb = std::min(ew.cap, n + 1 - k0);
    for (int b = 0; b < nb; ++b) {
      double* dst = ew.mats + count * b;
      if (k0 + b == 0) {
        ident_minus_f64_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(count, np, T0, dst);
        note_launch();
        RET(cudaGetLastError());
      } else {
        RET(load_Y(k0 + b - 1, dst));
      }
    }
    RET(logdet_spd(s, ew, mc, np, nb, ld + k0));
  }
  // Tr[D T0^(2j+1)] from S0 = T0^2, S2 = S0^2, S4 = S2^2, P1 = D T0, P3 = P1 S0
  EpiF64 e;
  RET(cudaMemsetAsync(tr, 0, 8 * sizeof(double), s));
  RET(launch_frob_dot(s, N, np, D, T0, fwork, tr + 0));                                    // Tr D T0
  if (nterms > 1) {
    RET(gemm_f64_nt(s, m, m, m, T0, np, T0, np, S, np, e, true));   // S0
    RET(gemm_f64_nt(s, m, m, m, D, np, T0, np, A1, np, e, false));   // P1 = D T0
    RET(launch_frob_dot(s, N, np, A1, S, fwork, tr + 1));                                   // Tr D T0^3
  }
  if (nterms > 2) {
    RET(gemm_f64_nt(s, m, m, m, S, np, S, np, Q, np, e, true));   // S2 = S0^2
    RET(launch_frob_dot(s, N, np, A1, Q, fwork, tr + 2));                                   // Tr D T0^5
  }
  if (nterms > 3) {
    RET(gemm_f64_nt(s, m, m, m, A1, np, S, np, Mt, np, e, false));   // P3 = P1 S0
    RET(launch_frob_dot(s, N, np, Mt, Q, fwork, tr + 3));                                   // Tr D T0^7
  }
  if (nterms > 4) {
    RET(gemm_f64_nt(s, m, m, m, Q, np, Q, np, Yw, np, e, true));   // S4
    RET(launch_frob_dot(s, N, np, A1, Yw, fwork, tr + 4));                                  // Tr D T0^9
  }
  if (nterms > 5) RET(launch_frob_dot(s, N, np, Mt, Yw, fwork, tr + 5));                    // Tr D T0^11
  EntW w{};
  w.nld = n + 1;
  w.w_ld[0] = std::ldexp(1.0, n_sq);
  for (int k = 0; k < n; ++k) w.w_ld[1 + k] = std::ldexp(1.0, n_sq - 1 - k);
  w.ntr = nterms;
  for (int j = 0; j < nterms; ++j) w.w_tr[j] = std::ldexp(1.0, n_sq + 1) / (2.0 * j + 1.0);
  w.cst = N * std::log(2.0);
  entropy_combine_kernel<<<1, 32, 0, s>>>(w, ld, tr, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_entropy_f64(cudaStream_t s, MatSet& m, EntropyWork& area, int N, double beta, int n_sq, double mu, double dmu,
                               const double* D, const double* H, double* work, double* out) {
  (void)beta;
  (void)mu;
  (void)dmu;
  (void)H;
  const size_t count = (size_t)m.np * m.np;
  auto load_Y = [&](int k, double* dst) {
    block_or_identity_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(count, N, m.np, m.Y[k], dst);
    note_launch();
    return cudaGetLastError();
  };
  return entropy_fp64(s, N, m.np, m.n, n_sq, m.T[0], load_Y, area, m.S, m.Q, m.Yw, m.A1, m.Mt, 6, D, work, out);
}

}  // namespace xl
