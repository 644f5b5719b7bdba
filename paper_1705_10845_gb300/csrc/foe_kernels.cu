// Element-wise and reduction kernels of the recursive Fermi-operator expansion
// and of its response chains (FP64 storage), plus the small FP64 vector
// algebra of the rank-m kernel update (Eqs. K_up, v_1; Woodbury form).
//
// The expansion is run in its tanh-doubling form: with
// T_0 = -beta (H - mu I) / 2^(n+1), the recursion
// X_{k+1} = X_k^2 [X_k^2 + (I - X_k)^2]^-1 on X = (I + T)/2 becomes
// T_{k+1} = 2 T_k (I + T_k^2)^-1 and D = (I + T_n)/2.
#include <algorithm>

#include "precision.h"

namespace xl {
namespace {

#define RET(x)                        \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

// Element-wise kernels over the leading m x m block of matrices with leading dimension np.
__global__ void t0_init_kernel(int n, int m, int np, const double* H, double mu, double scale,
                               double* T0) {
  grid_wait();
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (int)(e / m), j = (int)(e % m);
  if (i >= m) return;
  const size_t idx = (size_t)i * np + j;
  double v = 0.0;
  if (i < n && j < n) v = -scale * (H[idx] - (i == j ? mu : 0.0));
  T0[idx] = v;
}

__global__ void combine_kernel(int m, int np, double a, double c1, const double* X1, double c2,
                               const double* X2, double c3, const double* X3,
                               double* Y) {
  grid_wait();
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (int)(e / m), j = (int)(e % m);
  if (i >= m) return;
  const size_t idx = (size_t)i * np + j;
  double v = (i == j) ? a : 0.0;
  if (X1) v += c1 * X1[idx];
  if (X2) v += c2 * X2[idx];
  if (X3) v += c3 * X3[idx];
  Y[idx] = v;
}

// A1 = T0 diag(d) + diag(d) T0  (first level of a chain with diagonal T1_0)
__global__ void level0_A1_kernel(int m, int np, const double* T0, const double* d,
                                 double* A1) {
  grid_wait();
  const unsigned e = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = (int)(e / m), j = (int)(e % m);
  if (i >= m) return;
  const size_t idx = (size_t)i * np + j;
  A1[idx] = T0[idx] * (d[i] + d[j]);
}

// A1 = G + G^T through 32x32 shared-memory tiles (coalesced both ways; np is a multiple of 32).
__global__ void transpose_add_kernel(int np, const double* G, double* A1) {
  grid_wait();
  __shared__ double tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
  for (int r = ty; r < 32; r += 8) tile[r][tx] = G[(size_t)(bx + r) * np + by + tx];   // rows of block (bx, by)^T
  __syncthreads();
  for (int r = ty; r < 32; r += 8) {
    const size_t o = (size_t)(by + r) * np + bx + tx;
    A1[o] = G[o] + tile[tx][r];
  }
}

// out[i] = sum_{j < k} Y_ij M_ij (i < n): the diagonal of Y M^T, one warp per row.
__global__ void row_dot_kernel(int n, int k, int np, const double* Y, const double* M,
                               double* out) {
  grid_wait();
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;
  const double* y = Y + (size_t)i * np;
  const double* m = M + (size_t)i * np;
  double acc = 0.0;
  for (int j = lane; j < k; j += 32) acc += y[j] * m[j];
  acc = warp_sum(acc);
  if (lane == 0) out[i] = acc;
}

__global__ void get_diag_kernel(int n, int np, const double* X, double* out) {
  grid_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = X[(size_t)i * np + i];
}

__global__ void sum_kernel(int n, const double* __restrict__ x, double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += x[i];
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = acc;
}

// partial[b] = sum over rows b, b + gridDim.x, ... of sum_{j<n} A_ij B_ij
__global__ void frob_partial_kernel(int n, int np, const double* __restrict__ A, const double* __restrict__ B,
                                    double* __restrict__ partial) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int i = blockIdx.x; i < n; i += gridDim.x)
    for (int j = threadIdx.x; j < n; j += blockDim.x) acc += A[(size_t)i * np + j] * B[(size_t)i * np + j];
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) partial[blockIdx.x] = acc;
}

// ---- vector algebra of the response chains and of the rank-m kernel update ----
//
// Vectors of nat or 4 nat doubles, one block per system or probe and all of them in one launch: the
// work is nothing, a launch costs 2 to 3 us, and with 2 FP64 operations a clock on an SM a reduction
// over a block of 1024 threads takes 1.4 us by its shuffles alone.  So few threads and few reductions
// per block.  A probe of 96 atoms in a group of 48 took 8.2 us in sf_dot and gamma_apply, 7.8 us in
// the expansion and 8.6 us at the end.

constexpr int kVecThreads = 256;
constexpr int kMaxJobs = 16;

// The jobs of a launch travel in the kernel parameters.
template <class Job, int NJ>
struct JobList {
  int n = 0;
  Job job[NJ];
};

// sums of a and b over a block of kVecThreads; valid in every thread (sh: 16 doubles)
__device__ __forceinline__ void block_sum2(double& a, double& b, double* sh) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  a = warp_sum(a);
  b = warp_sum(b);
  __syncthreads();
  if (lane == 0) {
    sh[wid] = a;
    sh[8 + wid] = b;
  }
  __syncthreads();
  a = sh[lane & 7];
  b = sh[8 + (lane & 7)];
  for (int o = 4; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
}

// t = SF^T x per job: a block takes 32 of its kp structure factors
template <int NJ>
__global__ void __launch_bounds__(1024) probe_dot_kernel(const __grid_constant__ JobList<ProbeJob, NJ> L) {
  grid_wait();
  const ProbeJob& J = L.job[blockIdx.y];
  __shared__ double sh[32][33];
  const int c = threadIdx.x & 31, w = threadIdx.x >> 5, g = blockIdx.x * 32 + c;
  if (blockIdx.x * 32 >= J.kp) return;
  double acc = 0.0;
  if (g < J.kp) {
    const double *SF = J.SF, *x = J.x;
#pragma unroll 4
    for (int I = w; I < J.nat; I += 32) acc += SF[(size_t)I * J.kp + g] * x[I];
  }
  sh[w][c] = acc;
  __syncthreads();
  const int gw = blockIdx.x * 32 + w;   // warp w sums column w
  const double s = warp_sum(sh[c][w]);
  if (c == 0 && gw < J.kp) J.tmp[gw] = s;
}

// pot_I = sum_J gamma_real_IJ x_J + k sum_g SF[I][g] t[g], one block per row.  For a unit probe x = e_u
// the first sum is the element gamma_real_Iu and t is row u of SF.
template <int NJ>
__global__ void probe_apply_kernel(double k, const __grid_constant__ JobList<ProbeJob, NJ> L) {
  grid_wait();
  const ProbeJob& J = L.job[blockIdx.y];
  __shared__ double sh[32];
  const int I = blockIdx.x;
  if (I >= J.nat) return;
  double acc = 0.0, rec = 0.0;
  const double* gam = J.gam + (size_t)I * J.natp;
  if (J.unit >= 0) {
    if (threadIdx.x == 0) acc = gam[J.unit];
  } else {
    const double* x = J.x;
#pragma unroll 4
    for (int q = threadIdx.x; q < J.nat; q += blockDim.x) acc += gam[q] * x[q];
  }
  if (J.SF) {
    const double* row = J.SF + (size_t)I * J.kp;
    const double* t = (J.unit >= 0) ? J.SF + (size_t)J.unit * J.kp : J.tmp;
#pragma unroll 4
    for (int g = threadIdx.x; g < J.kp; g += blockDim.x) rec += row[g] * t[g];
  }
  acc = block_sum(acc + k * rec, sh);
  if (threadIdx.x == 0) J.pot[I] = acc;
}

// dvec_a = scale (pot_I - pbar) on the orbitals of atom I, 0 on the padding (one block per job).  A uniform
// potential has no canonical response (mu follows it); taking the average pbar = sum_a dmu_a pot_a /
// sum_a dmu_a out beforehand leaves sum_a d1_a = -sum_a pot_a dmu_a at rounding level, so that the
// chain does not carry a large part that mu_1 dT_n/dmu then has to cancel (the errors of the two are
// independent).  A unit probe's potential is mostly uniform: K of 48 atoms in FP16x3 was 2e-5 off
// without the shift.
// The chain runs on 2^-e dvec, |dvec| < 2^e its largest element, so that the scales of its operands have the
// same range to work in whatever the size of the probe; probe_finish_kernel takes d1 back by 2^e (scal[3]).
// Powers of two change no bit of w.  (At the probe's own size FP16 pairs lost w below |v| = 1e-17 and had NaN above 1e19.)
template <int NJ>
__global__ void __launch_bounds__(kVecThreads) probe_expand_kernel(double scale, const __grid_constant__ JobList<ProbeJob, NJ> L) {
  grid_wait();
  const ProbeJob& J = L.job[blockIdx.x];
  __shared__ double sh[16];
  const double *pot = J.pot, *dmu = J.dmu;
  double s0 = 0.0, s1 = 0.0;
  for (int a = threadIdx.x; a < 4 * J.nat; a += kVecThreads) {
    s0 += dmu[a];
    s1 += dmu[a] * pot[a >> 2];
  }
  block_sum2(s0, s1, sh);
  double pbar = s1 / s0;
  if (!isfinite(pbar)) pbar = 0.0;
  // the high words of |x| order like the numbers themselves
  __shared__ int top[kVecThreads / 32];
  int m = 0;
  for (int I = threadIdx.x; I < J.nat; I += kVecThreads) m = max(m, __double2hiint(fabs(scale * (pot[I] - pbar))));
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) top[threadIdx.x >> 5] = m;
  __syncthreads();
  m = __reduce_max_sync(0xffffffffu, top[threadIdx.x & (kVecThreads / 32 - 1)]);
  const int ex = m >> 20;   // biased exponent; 0 and 2047: nothing to scale
  const int e = (ex == 0 || ex == 2047) ? 0 : max(-900, min(ex - 1022, 900));
  const double f = scale * __hiloint2double((1023 - e) << 20, 0);   // scale 2^-e
  if (threadIdx.x == 0) J.scal[3] = __hiloint2double((1023 + e) << 20, 0);
  for (int I = threadIdx.x; I < J.nat; I += kVecThreads) {
    const double x = f * (pot[I] - pbar);
    for (int a = 4 * I; a < 4 * I + 4; ++a) J.dvec[a] = x;
  }
  for (int a = 4 * J.nat + threadIdx.x; a < J.np; a += kVecThreads) J.dvec[a] = 0.0;
}

// mu1 = -sum d1 / sum dmu;  w_I = sum_{a in I} (d1_a + mu1 dmu_a)  (one block per job), for the d1 of the
// scaled probe; the results are taken back by 2^e (up).  A unit probe's w - e_u is column u of J - I
// (row-major nat x nat at Jm), next to a column of the identity at B.
template <int NJ>
__global__ void __launch_bounds__(kVecThreads) probe_finish_kernel(const __grid_constant__ JobList<ProbeJob, NJ> L) {
  grid_wait();
  const ProbeJob& J = L.job[blockIdx.x];
  __shared__ double sh[16];
  const double *d1 = J.d1, *dmu = J.dmu;
  const double up = J.scal[3];
  double s1 = 0.0, s2 = 0.0;
  for (int a = threadIdx.x; a < J.N; a += kVecThreads) {
    s1 += d1[a];
    s2 += dmu[a];
  }
  block_sum2(s1, s2, sh);
  const double mu1 = (s2 != 0.0) ? -s1 / s2 : 0.0;
  if (threadIdx.x == 0) {
    J.scal[0] = s1 * up;
    J.scal[1] = s2;
    J.scal[2] = mu1 * up;
  }
  for (int I = threadIdx.x; I < J.nat; I += kVecThreads) {
    double t = 0.0;
    for (int a = 4 * I; a < 4 * I + 4; ++a) t += d1[a] + mu1 * dmu[a];
    t *= up;
    if (J.w) J.w[I] = t;
    if (J.unit >= 0) {
      const size_t o = (size_t)I * J.nat + J.unit;
      J.Jm[o] = t - (I == J.unit ? 1.0 : 0.0);
      J.B[o] = (I == J.unit) ? 1.0 : 0.0;
    }
  }
}

// out[q] = sum_{I < n} f(q, I) for q < cnt, a warp or several per sum (part: the block's warps x 1
// double, or cnt if that is more); valid in every thread after the call
template <class F>
__device__ __forceinline__ void block_dots(int cnt, int n, double* part, double* out, F f) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int split = cnt < nw ? nw / cnt : 1;
  for (int u = wid; u < cnt * split; u += nw) {
    const int q = u / split;
    double acc = 0.0;
    for (int I = (u % split) * 32 + lane; I < n; I += 32 * split) acc += f(q, I);
    acc = warp_sum(acc);
    if (lane == 0) part[u] = acc;
  }
  __syncthreads();
  if ((int)threadIdx.x < cnt) {
    double t = 0.0;
    for (int p = 0; p < split; ++p) t += part[threadIdx.x * split + p];
    out[threadIdx.x] = t;
  }
  __syncthreads();
}

// Rank-m kernel update, one block per system.
//
// With orthonormal probes V (rows), responses W, U = W - c V and
// S = (c - 1) I_m + V U^T, the Sherman-Morrison sequence of Eq. K_up equals
// K_m x = [x - U^T S^-1 V x] / (c - 1).
// mode 0: v_i = K_{i} r orthonormalised (two Gram-Schmidt passes) against the
//         first i probes; flag = 1 and V[i] = v_i, or flag = 0 when less than
//         1e-12 of it is left (K_i r already in the span).
// mode 1: out = K_m r.
// The m^2 + m sums of S and V r are taken side by side, as are the sums of a Gram-Schmidt pass (the
// classical form, twice), so that the chain of reductions does not grow with m.  One sum after the
// other by 1024 threads this took 17 us at m = 2 and 40 us at m = 4 for 512 atoms.
template <int NJ>
__global__ void __launch_bounds__(512) kernel_vec_kernel(const __grid_constant__ JobList<KernelVecJob, NJ> L) {
  grid_wait();
  const KernelVecJob& J = L.job[blockIdx.x];
  __shared__ double part[kMaxRank * (kMaxRank + 1)];
  __shared__ double dots[kMaxRank * (kMaxRank + 1)];
  const int tid = threadIdx.x, nat = J.nat, m = J.m;
  const double c = J.c;
  const double *r = J.r, *V = J.V, *W = J.W;
  double* x = (J.mode == 1) ? J.out : J.V + (size_t)m * nat;   // mode 0: the candidate goes to V[m]
  // x = K_m r
  if (m > 0) {
    const int ld = m + 1;
    block_dots(m * ld, nat, part, dots, [&](int q, int I) {
      const int a = q / ld, b = q % ld;
      const double va = V[(size_t)a * nat + I];
      return b == m ? va * r[I] : va * (W[(size_t)b * nat + I] - c * V[(size_t)b * nat + I]);
    });
    if (tid < m) dots[tid * ld + tid] += c - 1.0;
    __syncthreads();
    if (tid < 32) {
      // Gaussian elimination with partial pivoting on S y = V r, lane b at column b; y ends in column m
      for (int col = 0; col < m; ++col) {
        int piv = col;
        for (int a = col + 1; a < m; ++a)
          if (fabs(dots[a * ld + col]) > fabs(dots[piv * ld + col])) piv = a;
        __syncwarp();
        if (piv != col && tid <= m) {
          const double t = dots[col * ld + tid];
          dots[col * ld + tid] = dots[piv * ld + tid];
          dots[piv * ld + tid] = t;
        }
        __syncwarp();
        if (tid > col && tid <= m)
          for (int a = col + 1; a < m; ++a)
            dots[a * ld + tid] -= dots[a * ld + col] / dots[col * ld + col] * dots[col * ld + tid];
        __syncwarp();
      }
      for (int a = m - 1; a >= 0; --a) {
        const double y = dots[a * ld + m] / dots[a * ld + a];
        __syncwarp();
        if (tid < a) dots[tid * ld + m] -= dots[tid * ld + a] * y;
        if (tid == a) dots[a * ld + m] = y;
        __syncwarp();
      }
    }
    __syncthreads();
  }
  for (int I = tid; I < nat; I += blockDim.x) {
    double t = r[I];
    for (int a = 0; a < m; ++a) t -= (W[(size_t)a * nat + I] - c * V[(size_t)a * nat + I]) * dots[a * (m + 1) + m];
    x[I] = t / (c - 1.0);
  }
  if (J.mode == 1) return;
  __syncthreads();
  double n0 = 0.0;
  for (int pass = 0; pass < 2 && m > 0; ++pass) {
    // the first pass also takes |x|^2
    const int cnt = m + (pass == 0 ? 1 : 0);
    block_dots(cnt, nat, part, dots, [&](int q, int I) { return (q == m ? x[I] : V[(size_t)q * nat + I]) * x[I]; });
    if (pass == 0) n0 = sqrt(dots[m]);
    for (int I = tid; I < nat; I += blockDim.x) {
      double t = x[I];
      for (int a = 0; a < m; ++a) t -= dots[a] * V[(size_t)a * nat + I];
      x[I] = t;
    }
    __syncthreads();
  }
  block_dots(1, nat, part, dots, [&](int, int I) { return x[I] * x[I]; });
  const double nv = sqrt(dots[0]);
  if (m == 0) n0 = nv;
  const bool ok = (n0 > 0.0) && isfinite(nv) && (nv > 1e-12 * n0);
  if (ok)
    for (int I = tid; I < nat; I += blockDim.x) x[I] /= nv;
  if (tid == 0) *J.flag = ok ? 1.0 : 0.0;
}

// max |x_i|; any value that is not finite makes it NaN, so that the host sees it
__global__ void absmax_kernel(int n, const double* x, double* out) {
  grid_wait();
  __shared__ double sh[32];
  double m = 0.0;
  bool bad = false;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    bad |= !isfinite(x[i]);
    m = fmax(m, fabs(x[i]));
  }
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  bad = __syncthreads_or(bad);
  if (threadIdx.x < 32) {
    m = (threadIdx.x < (blockDim.x >> 5)) ? sh[threadIdx.x] : 0.0;
    m = warp_max(m);
    if (threadIdx.x == 0) *out = bad ? nan("") : m;
  }
}

__global__ void fill_history_kernel(int nat, int kmax, double* __restrict__ nh) {
  const int I = blockIdx.x * blockDim.x + threadIdx.x;
  if (I >= nat) return;
  for (int k = 1; k <= kmax; ++k) nh[(size_t)k * nat + I] = nh[I];
}

__global__ void axpy_kernel(int n, double a, const double* __restrict__ x, double* __restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] += a * x[i];
}

__global__ void diag_sum_kernel(int n, int np, const double* __restrict__ X, double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += X[(size_t)i * np + i];
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = acc;
}

// ddiag_a = 1 + Tn_aa + dmu Tmu_aa (a < N);  D = (I + Tn + dmu Tmu) / 2 on the N x N block, 0 elsewhere
__global__ void density_out_kernel(int N, int np, const double* __restrict__ Tn, const double* __restrict__ Tmu,
                                   double dmu, double* __restrict__ ddiag, double* __restrict__ D) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)np * np) return;
  const int i = (int)(idx / np), j = (int)(idx % np);
  double v = 0.0;
  if (i < N && j < N) {
    v = 0.5 * (Tn[idx] + dmu * Tmu[idx] + (i == j ? 1.0 : 0.0));
    if (i == j) ddiag[i] = 2.0 * v;
  }
  D[idx] = v;
}

inline unsigned blocks_for(size_t count, int tpb) { return (unsigned)((count + tpb - 1) / tpb); }

}  // namespace

namespace {

// f(list) with the jobs in lists of one, or of at most 16 (1.9 KB of parameters)
template <class Job, class F>
cudaError_t in_lists(const std::vector<Job>& jobs, F f) {
  if (jobs.size() == 1) {
    JobList<Job, 1> L;
    L.n = 1;
    L.job[0] = jobs[0];
    return f(L);
  }
  for (size_t i = 0; i < jobs.size(); i += kMaxJobs) {
    JobList<Job, kMaxJobs> L;
    L.n = (int)std::min<size_t>(kMaxJobs, jobs.size() - i);
    std::copy_n(jobs.begin() + i, L.n, L.job);
    RET(f(L));
  }
  return cudaSuccess;
}

template <int NJ>
cudaError_t probe_potential(cudaStream_t s, double k, JobList<ProbeJob, NJ>& L) {
  int nat = 0, dots = 0;
  for (int j = 0; j < L.n; ++j) {
    if (k == 0.0) L.job[j].SF = nullptr;
    nat = std::max(nat, L.job[j].nat);
    if (L.job[j].SF && L.job[j].unit < 0) dots = std::max(dots, L.job[j].kp);
  }
  if (dots) RET(launch_chained(s, dim3((dots + 31) / 32, L.n), 1024, 0, probe_dot_kernel<NJ>, L));
  // a row has nat + kp products
  return launch_chained(s, dim3(nat, L.n), nat <= 2048 ? 256 : 512, 0, probe_apply_kernel<NJ>, k, L);
}

template <int NJ>
cudaError_t kernel_vec(cudaStream_t s, const JobList<KernelVecJob, NJ>& L) {
  int nat = 0;
  for (int j = 0; j < L.n; ++j) nat = std::max(nat, L.job[j].nat);
  return launch_chained(s, L.n, nat <= 256 ? 256 : 512, 0, kernel_vec_kernel<NJ>, L);
}

template <int NJ>
cudaError_t probe_expand(cudaStream_t s, double scale, const JobList<ProbeJob, NJ>& L) {
  return launch_chained(s, L.n, kVecThreads, 0, probe_expand_kernel<NJ>, scale, L);
}

template <int NJ>
cudaError_t probe_finish(cudaStream_t s, const JobList<ProbeJob, NJ>& L) {
  return launch_chained(s, L.n, kVecThreads, 0, probe_finish_kernel<NJ>, L);
}

}  // namespace

cudaError_t launch_probe_potential(cudaStream_t s, double k, const std::vector<ProbeJob>& jobs) {
  return in_lists(jobs, [&](auto& L) { return probe_potential(s, k, L); });
}

cudaError_t launch_probe_expand(cudaStream_t s, double scale, const std::vector<ProbeJob>& jobs) {
  return in_lists(jobs, [&](auto& L) { return probe_expand(s, scale, L); });
}

cudaError_t launch_probe_finish(cudaStream_t s, const std::vector<ProbeJob>& jobs) {
  return in_lists(jobs, [&](auto& L) { return probe_finish(s, L); });
}

cudaError_t launch_kernel_vec(cudaStream_t s, const std::vector<KernelVecJob>& jobs) {
  return in_lists(jobs, [&](auto& L) { return kernel_vec(s, L); });
}

cudaError_t launch_absmax(cudaStream_t s, int n, const double* x, double* out) {
  return launch_chained(s, 1, 256, 0, absmax_kernel, n, x, out);
}

cudaError_t launch_fill_history(cudaStream_t s, int nat, int kmax, double* nh) {
  fill_history_kernel<<<blocks_for(nat, 128), 128, 0, s>>>(nat, kmax, nh);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_axpy(cudaStream_t s, int n, double a, const double* x, double* y) {
  axpy_kernel<<<blocks_for(n, 128), 128, 0, s>>>(n, a, x, y);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_diag_sum(cudaStream_t s, int n, int np, const double* X, double* out) {
  diag_sum_kernel<<<1, 1024, 0, s>>>(n, np, X, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_density_out_f64(cudaStream_t s, int N, int np, const double* Tn, const double* Tmu, double dmu,
                                   double* ddiag, double* D) {
  density_out_kernel<<<blocks_for((size_t)np * np, 256), 256, 0, s>>>(N, np, Tn, Tmu, dmu, ddiag, D);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_t0_init(cudaStream_t s, int n, int m, int np, const double* H, double mu, double scale, double* T0) {
  RET(launch_chained(s, blocks_for((size_t)m * m, 256), 256, 0, t0_init_kernel, n, m, np, H, mu, scale, T0));
  return cudaSuccess;
}

cudaError_t launch_combine(cudaStream_t s, int m, int np, double a, double c1, const double* X1, double c2,
                           const double* X2, double c3, const double* X3, double* Y) {
  RET(launch_chained(s, blocks_for((size_t)m * m, 256), 256, 0, combine_kernel, m, np, a, c1, X1, c2, X2, c3, X3, Y));
  return cudaSuccess;
}

cudaError_t launch_level0_A1(cudaStream_t s, int m, int np, const double* T0, const double* d, double* A1) {
  RET(launch_chained(s, blocks_for((size_t)m * m, 256), 256, 0, level0_A1_kernel, m, np, T0, d, A1));
  return cudaSuccess;
}

cudaError_t launch_transpose_add(cudaStream_t s, int m, int np, const double* G, double* A1) {
  if (np % 32) return cudaErrorInvalidValue;
  dim3 grid((m + 31) / 32, (m + 31) / 32), block(32, 8);
  RET(launch_chained(s, grid, block, 0, transpose_add_kernel, np, G, A1));
  return cudaSuccess;
}

cudaError_t launch_row_dot(cudaStream_t s, int n, int k, int np, const double* Y, const double* M, double* out) {
  RET(launch_chained(s, (n + 7) / 8, 256, 0, row_dot_kernel, n, k, np, Y, M, out));
  return cudaSuccess;
}

cudaError_t launch_get_diag(cudaStream_t s, int n, int np, const double* X, double* out) {
  RET(launch_chained(s, (n + 255) / 256, 256, 0, get_diag_kernel, n, np, X, out));
  return cudaSuccess;
}

cudaError_t launch_sum(cudaStream_t s, int n, const double* x, double* out) {
  sum_kernel<<<1, 1024, 0, s>>>(n, x, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_frob_dot(cudaStream_t s, int n, int np, const double* A, const double* B, double* work,
                            double* out) {
  const int nb = n < 1024 ? n : 1024;
  frob_partial_kernel<<<nb, 256, 0, s>>>(n, np, A, B, work);
  note_launch();
  sum_kernel<<<1, 1024, 0, s>>>(nb, work, out);
  note_launch();
  return cudaGetLastError();
}

// ---- exact kernel K = (J - I)^-1 (Eq. KK) ----

namespace {

// In-place Gauss-Jordan inverse with partial pivoting of a matrix that fits the shared memory of one
// cluster: column j lives in CTA j mod 8, one warp per column.  Per step the warp that holds the pivot
// column searches it and sends the row exchange, 1/pivot and the factors to all CTAs; every warp then
// updates its own columns, and the next pivot column goes first, so that its search and the cluster
// barrier run beside the rest of the update.  The factors are held three deep: a CTA arrives for step k + 1
// when it enters step k, done with k - 1.  At n = 96 the update's FP64 work is 0.3 us a step (a CTA has 2
// FMAs a clock); the 2.5 us a step that were measured (237 us in all; as a search and an elimination
// launch per step 1340) are the chain of search, division, remote stores and cluster barrier.
constexpr int kGjCtas = 8, kGjThreads = 512, kGjMaxSmem = 227 * 1024;

__host__ __device__ inline size_t gj_smem(int n) {
  const size_t cols = (n + kGjCtas - 1) / kGjCtas;
  return sizeof(double) * (cols * (n | 1) + 3 * (size_t)(n + 2)) + 3 * sizeof(int) * (size_t)n;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ void st_cluster(uint32_t addr, uint32_t cta, double v) {
  uint32_t remote;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(addr), "r"(cta));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(remote), "d"(v) : "memory");
}

__global__ void __cluster_dims__(kGjCtas, 1, 1) __launch_bounds__(kGjThreads)
    gj_cluster_kernel(int n, const double* __restrict__ A, double* __restrict__ B, double* __restrict__ flag) {
  extern __shared__ double sm[];
  const int cta = blockIdx.x, lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = kGjThreads / 32;
  const int cols = (n - cta + kGjCtas - 1) / kGjCtas, ld = n | 1;
  double* fs = sm + (size_t)((n + kGjCtas - 1) / kGjCtas) * ld;   // 3 x [n factors, 1/pivot, pivot row]
  int* piv = reinterpret_cast<int*>(fs + 3 * (n + 2));
  int *src = piv + n, *dst = src + n;
  for (int e = threadIdx.x; e < n * cols; e += kGjThreads) {
    const int i = e / cols, c = e % cols;
    sm[(size_t)c * ld + i] = A[(size_t)i * n + cta + kGjCtas * c];
  }
  __syncthreads();
  cluster_arrive();   // every CTA has started before the first remote store
  cluster_wait();

  // one warp: pivot search of column k in rows k .. n - 1, its exchange, factors and inverse column
  auto publish = [&](int k) {
    double* col = sm + (size_t)(k / kGjCtas) * ld;
    double best = -1.0;
    int p = k;
    for (int i = k + lane; i < n; i += 32) {
      const double v = fabs(col[i]);
      if (v > best) {
        best = v;
        p = i;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int op = __shfl_xor_sync(0xffffffffu, p, o);
      if (ov > best || (ov == best && op < p)) {
        best = ov;
        p = op;
      }
    }
    const double pv = col[p], top = col[k];
    const bool bad = !(fabs(pv) > 0.0) || !isfinite(pv);
    const double inv = bad ? 0.0 : 1.0 / pv;
    __syncwarp();
    const uint32_t f = (uint32_t)__cvta_generic_to_shared(fs + (size_t)(k % 3) * (n + 2));
    for (int i = lane; i < n; i += 32) {
      const double v = (i == k) ? 0.0 : (i == p) ? top : col[i];
      for (int c = 0; c < kGjCtas; ++c) st_cluster(f + 8 * i, c, v);
      col[i] = (i == k) ? inv : -v * inv;
    }
    if (lane < kGjCtas) {
      st_cluster(f + 8 * n, lane, inv);
      st_cluster(f + 8 * (n + 1), lane, (double)p);
    }
    __syncwarp();
  };

  if (cta == 0 && wid == 0) publish(0);
  cluster_arrive();
  bool bad = false;
  for (int k = 0; k < n; ++k) {
    cluster_wait();
    const double* f = fs + (size_t)(k % 3) * (n + 2);
    const double inv = f[n];
    const int p = (int)f[n + 1];
    if (inv == 0.0) {   // the same in every thread of the cluster
      bad = true;
      break;
    }
    if (threadIdx.x == 0) piv[k] = p;
    auto update = [&](int c) {
      double* col = sm + (size_t)c * ld;
      const double top = col[k], ck = col[p] * inv;
      __syncwarp();
      for (int i = lane; i < n; i += 32) {
        const double v = (i == p) ? top : col[i];
        col[i] = (i == k) ? ck : v - f[i] * ck;
      }
      __syncwarp();
    };
    const int next = (k + 1 < n && (k + 1) % kGjCtas == cta) ? (k + 1) / kGjCtas : -1;
    if (next >= 0 && next % nw == wid) {
      update(next);
      publish(k + 1);
    }
    if (k + 1 < n) cluster_arrive();
    for (int c = wid; c < cols; c += nw)
      if (c != next && cta + kGjCtas * c != k) update(c);
  }
  __syncthreads();
  if (!bad) {
    // the result is the inverse of the row-permuted matrix: undo the exchanges on its columns
    for (int j = threadIdx.x; j < n; j += kGjThreads) src[j] = j;
    __syncthreads();
    if (threadIdx.x == 0)
      for (int k = n - 1; k >= 0; --k) {
        const int p = piv[k], t = src[k];
        src[k] = src[p];
        src[p] = t;
      }
    __syncthreads();
    for (int j = threadIdx.x; j < n; j += kGjThreads) dst[src[j]] = j;
    __syncthreads();
    for (int e = threadIdx.x; e < n * cols; e += kGjThreads) {
      const int i = e / cols, c = e % cols;
      B[(size_t)i * n + dst[cta + kGjCtas * c]] = sm[(size_t)c * ld + i];
    }
  } else if (cta == 0 && threadIdx.x == 0) {
    *flag = 1.0;
  }
  cluster_arrive();   // no CTA leaves while another may still store into it
  cluster_wait();
}

// Gauss-Jordan step k, part 1 (one CTA): partial pivot of column k over rows k..n-1,
// swap of rows k and p in A and B, scaling of row k by 1 / A_kk, and the elimination
// factors f_i = A_ik (f_k = 0) copied out so that part 2 reads no column it writes.
__global__ void gj_pivot_kernel(int n, int k, double* __restrict__ A, double* __restrict__ B,
                                double* __restrict__ f, double* __restrict__ flag) {
  __shared__ double sv[32];
  __shared__ int si[32];
  __shared__ int s_p;
  double best = -1.0;
  int bi = k;
  for (int i = k + threadIdx.x; i < n; i += blockDim.x) {
    const double v = fabs(A[(size_t)i * n + k]);
    if (v > best) {
      best = v;
      bi = i;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > best || (ov == best && oi < bi)) {
      best = ov;
      bi = oi;
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    sv[wid] = best;
    si[wid] = bi;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double b = -1.0;
    int p = k;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w)
      if (sv[w] > b || (sv[w] == b && si[w] < p)) {
        b = sv[w];
        p = si[w];
      }
    s_p = p;
  }
  __syncthreads();
  const int p = s_p;
  if (p != k)
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      const double ta = A[(size_t)k * n + j], tb = B[(size_t)k * n + j];
      A[(size_t)k * n + j] = A[(size_t)p * n + j];
      B[(size_t)k * n + j] = B[(size_t)p * n + j];
      A[(size_t)p * n + j] = ta;
      B[(size_t)p * n + j] = tb;
    }
  __syncthreads();
  const double piv = A[(size_t)k * n + k];
  const bool bad = !(fabs(piv) > 0.0) || !isfinite(piv);
  __syncthreads();   // every thread has read the pivot before row k is scaled
  if (bad) {
    if (threadIdx.x == 0) *flag = 1.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) f[i] = 0.0;
    return;
  }
  const double inv = 1.0 / piv;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    A[(size_t)k * n + j] *= inv;
    B[(size_t)k * n + j] *= inv;
  }
  for (int i = threadIdx.x; i < n; i += blockDim.x) f[i] = (i == k) ? 0.0 : A[(size_t)i * n + k];
}

// Gauss-Jordan step k, part 2: row_i -= f_i row_k for every i != k, over A's columns >= k
// (the columns left of k are already those of the identity) and all of B's.
__global__ void gj_eliminate_kernel(int n, int k, double* __restrict__ A, double* __restrict__ B,
                                    const double* __restrict__ f) {
  const int i = blockIdx.y;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == k || j >= 2 * n) return;
  const double fi = f[i];
  if (fi == 0.0) return;
  if (j < n) {
    if (j >= k) A[(size_t)i * n + j] -= fi * A[(size_t)k * n + j];
  } else {
    const int c = j - n;
    B[(size_t)i * n + c] -= fi * B[(size_t)k * n + c];
  }
}

}  // namespace

cudaError_t launch_gauss_jordan(cudaStream_t s, int n, double* A, double* B, double* f, double* flag) {
  if (n < 1 || n > 65535) return cudaErrorInvalidValue;
  if (gj_smem(n) <= kGjMaxSmem) {   // n <= 463
    RET(cudaFuncSetAttribute(gj_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGjMaxSmem));
    gj_cluster_kernel<<<kGjCtas, kGjThreads, gj_smem(n), s>>>(n, A, B, flag);
    note_launch();
    return cudaGetLastError();
  }
  const dim3 grid((2 * n + 255) / 256, n);
  for (int k = 0; k < n; ++k) {
    gj_pivot_kernel<<<1, 1024, 0, s>>>(n, k, A, B, f, flag);
    note_launch();
    gj_eliminate_kernel<<<grid, 256, 0, s>>>(n, k, A, B, f);
    note_launch();
  }
  return cudaGetLastError();
}


// ---- accumulated rank-1 kernel (one Sherman-Morrison update per step) ----

namespace {

__global__ void scaled_identity_kernel(int n, double a, double* __restrict__ M) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * n) return;
  M[idx] = (idx / n == idx % n) ? a : 0.0;
}

// y_j = sum_i M_ij x_i (row-major n x n; one thread per column, coalesced over j)
__global__ void gemv_t_kernel(int n, const double* __restrict__ M, const double* __restrict__ x,
                              double* __restrict__ y) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  double acc = 0.0;
  for (int i = 0; i < n; ++i) acc += M[(size_t)i * n + j] * x[i];
  y[j] = acc;
}

// v <- v / |v|; flag = 1 when |v| is positive and finite, else 0 (v untouched)
__global__ void normalize_kernel(int n, double* __restrict__ v, double* __restrict__ flag) {
  __shared__ double sh[32];
  double a = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) a += v[i] * v[i];
  a = sqrt(block_sum(a, sh));
  const bool ok = a > 0.0 && isfinite(a);
  if (ok)
    for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] /= a;
  if (threadIdx.x == 0) *flag = ok ? 1.0 : 0.0;
}

// u = w - t;  out = 1 + v . Ku is formed later by dot1p_kernel
__global__ void sub_kernel(int n, const double* __restrict__ w, const double* __restrict__ t, double* __restrict__ u) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) u[i] = w[i] - t[i];
}

__global__ void dot1p_kernel(int n, const double* __restrict__ a, const double* __restrict__ b,
                             double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += a[i] * b[i];
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = 1.0 + acc;
}

// J += u v^T;  K -= (K u)(v^T K) / (1 + v^T K u)
__global__ void rank1_update_kernel(int n, const double* __restrict__ u, const double* __restrict__ v,
                                    const double* __restrict__ Ku, const double* __restrict__ vK,
                                    const double* __restrict__ denom, double* __restrict__ J, double* __restrict__ K) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * n) return;
  const int i = (int)(idx / n), j = (int)(idx % n);
  J[idx] += u[i] * v[j];
  K[idx] -= Ku[i] * vK[j] / *denom;
}

inline unsigned blocks_for(size_t count) { return (unsigned)((count + 255) / 256); }

}  // namespace

cudaError_t launch_scaled_identity(cudaStream_t s, int n, double a, double* M) {
  scaled_identity_kernel<<<blocks_for((size_t)n * n), 256, 0, s>>>(n, a, M);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_gemv_t(cudaStream_t s, int n, const double* M, const double* x, double* y) {
  gemv_t_kernel<<<blocks_for(n), 256, 0, s>>>(n, M, x, y);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_normalize(cudaStream_t s, int n, double* v, double* flag) {
  normalize_kernel<<<1, 1024, 0, s>>>(n, v, flag);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_sub(cudaStream_t s, int n, const double* w, const double* t, double* u) {
  sub_kernel<<<blocks_for(n), 256, 0, s>>>(n, w, t, u);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_dot1p(cudaStream_t s, int n, const double* a, const double* b, double* out) {
  dot1p_kernel<<<1, 1024, 0, s>>>(n, a, b, out);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_rank1_update(cudaStream_t s, int n, const double* u, const double* v, const double* Ku,
                                const double* vK, const double* denom, double* J, double* K) {
  rank1_update_kernel<<<blocks_for((size_t)n * n), 256, 0, s>>>(n, u, v, Ku, vK, denom, J, K);
  note_launch();
  return cudaGetLastError();
}

}  // namespace xl
