// Split-precision engine: the expansion and response chains with tensor-core
// products on hi/lo operand pairs (FP16x3, BF16x3 or TF32x3).
//
// Every matrix keeps a value array -- FP32, or double-float (an FP32 hi + lo
// pair) for T_k, M and T1, whose leading terms the correction form keeps out of
// the products -- and a split operand pair hi = rn(x s), lo = rn(x s - hi)
// (rn: rounding to FP16, BF16 or TF32).  The power-of-two scale s comes from a
// bound that is known before the matrix is computed (operand.cuh): |T_k| <= t_k
// from the spectral bound and the scalar recursion, everything that only
// matters against the identity below 4, and the chains' matrices, which are
// linear in the probe, from max |dvec| and the recursion's growth.  So every
// kernel that computes a matrix writes its operands in the same pass.  (The
// scales used to follow each matrix's own maximum: a memset, an atomic maximum
// and a conversion pass per product.)  A product takes three tensor-core
// products (hi*hi, hi*lo, lo*hi), or one (hi*hi) in the probe chains and
// dT_n/dmu when the context asks for it.  Traces, charges and the density
// matrix handed to the forces are accumulated in FP64.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <unordered_map>

#include "operand.cuh"
#include "precision.h"
#include "tc.h"

namespace xl {
namespace {

#define RET(x)                        \
  do {                                \
    cudaError_t e_ = (x);             \
    if (e_ != cudaSuccess) return e_; \
  } while (0)

inline unsigned nblk(size_t count, int tpb = 256) { return (unsigned)((count + tpb - 1) / tpb); }

// element-wise kernels walk their elements grid-stride with at most this many blocks
constexpr unsigned kEwBlocks = 152 * 16;

// One-CTA-per-tile product kernel: products of at least this size split their hi*hi sums over
// both accumulators.
constexpr int kSplitAccMin = 8192;
// Split products accumulate the hi*hi sum in chunks of K = 512 (8 K blocks of 64 16-bit or 16 of 32 TF32
// elements), added up with round-to-nearest FP32 adds.  The tensor core truncates as it accumulates, so a
// sum's error grows with its length: at 2048 atoms (N = 8192) the charge error fell from 4.7e-5 e (one
// 8192-long sum) to 2.5e-5 e (two halves) and 6.6e-6 e (1024-long chunks).  Product errors and times at
// n = 8192 for chunks of 256, 512, 1024 and the whole sum: 9e-5, 1.4e-4, 2.4e-4, 2e-3 and 2.83, 2.30, 2.21,
// 2.14 ms; at n = 1024 (128-wide tiles) 3e-5, 5e-5, 1e-4 and 29, 29, 28 us.
constexpr int kChunkK = 512;

// Operands of four values at element i in the format fmt (0 FP16, 1 BF16, 2 TF32).
__device__ __forceinline__ void store_op4(int fmt, void* hi, void* lo, size_t i, float s, const float (&x)[4],
                                          const float (&xl)[4]) {
  if (fmt == 2)
    store_operand4<2>(hi, lo, i, s, x, xl);
  else if (fmt == 1)
    store_operand4<1>(hi, lo, i, s, x, xl);
  else
    store_operand4<0>(hi, lo, i, s, x, xl);
}

__global__ void df_to_f64_kernel(size_t count, const float2* __restrict__ x, double* __restrict__ y) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) y[i] = (double)x[i].x + (double)x[i].y;
}

// dst = I - W on the N x N block (W an FP32 value, dst FP64), the identity around it: on the padding's
// diagonal W is what the corrections leave at eigenvalue zero, the same in every row (33 atoms with 14
// squarings: 60 rows put 1.5e-4 eV on the entropy)
__global__ void ident_minus_f32_to_f64_kernel(size_t count, int N, int np, const float* __restrict__ W,
                                              double* __restrict__ dst) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int r = (int)(i / np), c = (int)(i % np);
  dst[i] = (r == c ? 1.0 : 0.0) - (r < N && c < N ? (double)W[i] : 0.0);
}

__device__ __forceinline__ double df_val(float2 v) { return (double)v.x + (double)v.y; }

__global__ void diag_sum_d_kernel(int n, int np, const float2* __restrict__ X, double* __restrict__ out) {
  __shared__ double sh[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += df_val(X[(size_t)i * np + i]);
  acc = block_sum(acc, sh);
  if (threadIdx.x == 0) *out = acc;
}

__global__ void density_out_d_kernel(int N, int np, const float2* __restrict__ Tn, const float2* __restrict__ Tmu,
                                     double dmu, double* __restrict__ ddiag, double* __restrict__ D) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)np * np) return;
  const int i = (int)(idx / np), j = (int)(idx % np);
  double v = 0.0;
  if (i < N && j < N) {
    v = 0.5 * (df_val(Tn[idx]) + dmu * df_val(Tmu[idx]) + (i == j ? 1.0 : 0.0));
    if (i == j) ddiag[i] = 2.0 * v;
  }
  D[idx] = v;
}

// ---- grouped element-wise kernels ----
//
// Batched trajectories step in lockstep: the same element-wise operation runs on the matrices
// of every system of a group in one launch, blockIdx.y selecting the system.  The per-system
// pointers travel by value in the kernel parameters (at most kMaxGroup systems per launch).
constexpr int kMaxGroup = 64;

// Y = g0 I + g1 X1 + g2 X2 + g3 X3 per system (matrices not given are left out): the start of a level's
// inverse, and the sums of its corrections
struct CombList {
  int n = 0;
  const float* X[3][kMaxGroup];   // may be Y itself
  float* Y[kMaxGroup];
  void* hi[kMaxGroup];            // operands (lo: null for single products)
  void* lo[kMaxGroup];
  const float* scale[kMaxGroup];
  float g[4][kMaxGroup];
  const double* dg[kMaxGroup];   // device g when not null
};

__global__ void combine_group_kernel(int np, int fmt, CombList L) {
  grid_wait();
  const int j = blockIdx.y;
  float g[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) g[q] = L.dg[j] ? (float)L.dg[j][q] : L.g[q][j];
  const size_t count = (size_t)np * np / 4;
  const float4* X0 = reinterpret_cast<const float4*>(L.X[0][j]);
  const float4* X1 = reinterpret_cast<const float4*>(L.X[1][j]);
  const float4* X2 = reinterpret_cast<const float4*>(L.X[2][j]);
  float4* Y = reinterpret_cast<float4*>(L.Y[j]);
  const float s = *L.scale[j];
  const float zero[4] = {0.f, 0.f, 0.f, 0.f};
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < count; idx += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(4 * idx / np), c = (int)(4 * idx % np);   // np is a multiple of 4: one row
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    const float4* Xs[3] = {X0, X1, X2};
#pragma unroll
    for (int q = 0; q < 3; ++q)
      if (Xs[q]) {
        const float4 x = Xs[q][idx];
        v[0] += g[q + 1] * x.x;
        v[1] += g[q + 1] * x.y;
        v[2] += g[q + 1] * x.z;
        v[3] += g[q + 1] * x.w;
      }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (r == c + q) v[q] += g[0];
    Y[idx] = make_float4(v[0], v[1], v[2], v[3]);
    store_op4(fmt, L.hi[j], L.lo[j], 4 * idx, s, v, zero);
  }
}

// T0 = -sc (H - mu I) as a double-float with its operands, per system; the first thread also writes the
// operand scales of T_0 .. T_n (|T_k| <= t_k, t_{k+1} = 2 t_k / (1 + t_k^2)) and t_0 for the chains.
// mu and t_0 come from the device parameters dpar of a captured pass (dpar[0], dpar[dt0]) when given.
struct T0List {
  int n = 0;
  int N[kMaxGroup];
  const double* H[kMaxGroup];
  double mu[kMaxGroup];
  double t0[kMaxGroup];
  const double* dpar[kMaxGroup];
  float2* T0[kMaxGroup];
  void* hi[kMaxGroup];
  void* lo[kMaxGroup];
  float* scales[kMaxGroup];
  float* t0_dev[kMaxGroup];
};

__global__ void t0_init_group_kernel(int np, int nlev, int fmt, int dt0, double sc, T0List L) {
  grid_wait();
  const int j = blockIdx.y;
  const double mu = L.dpar[j] ? L.dpar[j][0] : L.mu[j];
  const double t0 = L.dpar[j] ? L.dpar[j][dt0] : L.t0[j];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    float* scales = L.scales[j];
    float t = (float)t0;   // FP32 for the same reason as in chain_scales_kernel
    scales[1] = operand_scale(t0);
    for (int k = 1; k <= nlev; ++k) {
      t = 2.0f * t / (1.0f + t * t);
      scales[1 + k] = operand_scale(t);
    }
    scales[2 + nlev] = operand_scale(1.0 / (1.0 - t0 * t0));   // |(I - T_0^2)^-1|
    *L.t0_dev[j] = (float)t0;
  }
  const float s = operand_scale(t0);
  const int n = L.N[j];
  const double* H = L.H[j];
  float2* T0 = L.T0[j];
  const size_t count = (size_t)np * np / 4;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < count; idx += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(4 * idx / np), c = (int)(4 * idx % np);
    const double2 a = reinterpret_cast<const double2*>(H)[2 * idx], b = reinterpret_cast<const double2*>(H)[2 * idx + 1];
    const double h[4] = {a.x, a.y, b.x, b.y};
    float x[4], xl[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      double v = 0.0;
      if (r < n && c + q < n) v = -sc * (h[q] - (r == c + q ? mu : 0.0));
      x[q] = (float)v;
      xl[q] = (float)(v - (double)x[q]);
    }
    float4* d = reinterpret_cast<float4*>(T0) + 2 * idx;
    d[0] = make_float4(x[0], xl[0], x[1], xl[1]);
    d[1] = make_float4(x[2], xl[2], x[3], xl[3]);
    store_op4(fmt, L.hi[j], L.lo[j], 4 * idx, s, x, xl);
  }
}

// Operand scales of a response chain, one block per system.  With tau_k a bound of |T1_k|
// (tau_0 = max |d|, T1_0 = diag(d)):
//   A1 = T T1 + T1 T           |A1| <= 2 t tau
//   M  = 2 T1 - A1 T'          |M|  <= 2 tau (1 + t t')
//   T1' = 2 Y (T1 - T T1 T) Y  |T1'| <= 2 tau (1 + g^2),  g = t / (1 + t^2) the largest t y
// Two-step chain: P = Y T1 in the place of M, |P| <= tau, and Q = T' T1 / 4 in that of A1 at the scale that
// makes Q T' match P W in one accumulator; |Q| times it stays below 2^14.
struct ChainScaleList {
  int n = 0;
  const double* d[kMaxGroup];
  const float* t0[kMaxGroup];
  const float* ts[kMaxGroup];   // two-step chain: the scales of T_0, T_1, ..  (null: three-step)
  float* scales[kMaxGroup];     // [3 k] A1_k, [3 k + 1] M_k, [3 k + 2] T1_{k+1}
};

__global__ void chain_scales_kernel(int np, int nlev, ChainScaleList L) {
  grid_wait();
  __shared__ float sm[32];
  const int j = blockIdx.x;
  float m = 0.0f;
  for (int i = threadIdx.x; i < np; i += blockDim.x) m = fmaxf(m, fabsf((float)L.d[j][i]));
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = fmaxf(m, sm[w]);
  // bounds slightly above the FP32 maximum, so that rounding them down cannot matter; in FP32, since one
  // thread's chain of FP64 divisions took 15 us at 12 levels
  float tau = 1.0001f * m, t = 1.0001f * *L.t0[j];
  float* scales = L.scales[j];
  for (int k = 0; k < nlev; ++k) {
    const float g = t / (1.0f + t * t), tn = 2.0f * g;
    const float* ts = L.ts[j];
    const float sp = ts ? operand_scale(tau) : operand_scale(2.0f * tau * (1.0f + t * tn));
    scales[3 * k] = ts ? sp * kUnitScale / ts[k + 1] : operand_scale(2.0f * t * tau);
    scales[3 * k + 1] = sp;
    tau *= 2.0f * (1.0f + g * g);
    scales[3 * k + 2] = operand_scale(tau);
    t = tn;
  }
}

// Operands of A1 = (T0 hi + lo)(d_i + d_j), chain level 0, per system (the value itself is not needed)
struct A1List {
  int n = 0;
  const float2* T0[kMaxGroup];
  const double* d[kMaxGroup];
  void* hi[kMaxGroup];
  void* lo[kMaxGroup];
  const float* scale[kMaxGroup];
};

__global__ void level0_A1_group_kernel(int np, int fmt, A1List L) {
  grid_wait();
  const int j = blockIdx.y;
  const float4* T0 = reinterpret_cast<const float4*>(L.T0[j]);
  const double* d = L.d[j];
  const float s = *L.scale[j];
  const float zero[4] = {0.f, 0.f, 0.f, 0.f};
  const size_t count = (size_t)np * np / 4;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < count; idx += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(4 * idx / np), c = (int)(4 * idx % np);
    const float4 a = T0[2 * idx], b = T0[2 * idx + 1];
    const double dr = d[r];
    const float x[4] = {(a.x + a.y) * (float)(dr + d[c]), (a.z + a.w) * (float)(dr + d[c + 1]),
                        (b.x + b.y) * (float)(dr + d[c + 2]), (b.z + b.w) * (float)(dr + d[c + 3])};
    store_op4(fmt, L.hi[j], L.lo[j], 4 * idx, s, x, zero);
  }
}

// Two-step chain, level 0, per system: P = (I - W) diag(d) and Q = T' diag(d) / 4, value and operands
struct P0List {
  int n = 0;
  const float* W[kMaxGroup];
  const float2* T[kMaxGroup];
  const double* d[kMaxGroup];
  float* Pf[kMaxGroup];    // P as FP32 (single products) ..
  float2* Pd[kMaxGroup];   // .. or as double-float
  float* Qf[kMaxGroup];
  void *Phi[kMaxGroup], *Plo[kMaxGroup], *Qhi[kMaxGroup], *Qlo[kMaxGroup];
  const float *Ps[kMaxGroup], *Qs[kMaxGroup];
};

__global__ void level0_P_group_kernel(int np, int fmt, P0List L) {
  grid_wait();
  const int j = blockIdx.y;
  const float4* W = reinterpret_cast<const float4*>(L.W[j]);
  const float4* T = reinterpret_cast<const float4*>(L.T[j]);
  const double* d = L.d[j];
  const float sp = *L.Ps[j], sq = *L.Qs[j];
  const float zero[4] = {0.f, 0.f, 0.f, 0.f};
  const size_t count = (size_t)np * np / 4;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < count; idx += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(4 * idx / np), c = (int)(4 * idx % np);
    const float4 w4 = W[idx], a = T[2 * idx], b = T[2 * idx + 1];
    const float w[4] = {w4.x, w4.y, w4.z, w4.w}, t[4] = {a.x + a.y, a.z + a.w, b.x + b.y, b.z + b.w};
    float p[4], pl[4], q[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const double dc = d[c + e], v = ((r == c + e ? 1.0 : 0.0) - (double)w[e]) * dc;
      p[e] = (float)v;
      pl[e] = (float)(v - (double)p[e]);
      q[e] = 0.25f * t[e] * (float)dc;
    }
    if (L.Pf[j]) {
      reinterpret_cast<float4*>(L.Pf[j])[idx] = make_float4(p[0], p[1], p[2], p[3]);
    } else {
      float4* o = reinterpret_cast<float4*>(L.Pd[j]) + 2 * idx;
      o[0] = make_float4(p[0], pl[0], p[1], pl[1]);
      o[1] = make_float4(p[2], pl[2], p[3], pl[3]);
    }
    reinterpret_cast<float4*>(L.Qf[j])[idx] = make_float4(q[0], q[1], q[2], q[3]);
    store_op4(fmt, L.Phi[j], L.Plo[j], 4 * idx, sp, p, pl);
    store_op4(fmt, L.Qhi[j], L.Qlo[j], 4 * idx, sq, q, zero);
  }
}

// Diagonal reductions of the chains' last level, per system
struct DiagList {
  int n = 0;
  int N[kMaxGroup];
  const float* W[kMaxGroup];    // row_dot: W_k (FP32)
  const float2* X[kMaxGroup];   // row_dot: M^T, or P; get_diag: T1_n (double-float)
  const float* Q[kMaxGroup];    // two-step chain: Q and T'
  const float2* T[kMaxGroup];
  double* out[kMaxGroup];
};

// out_i = T1'_ii = 2 P_ii - 2 sum_j (P_ij W_ij + Q_ij T'_ij), one warp per row
__global__ void row_dot_two_group_kernel(int np, DiagList L) {
  grid_wait();
  const int j = blockIdx.y;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= L.N[j]) return;
  const size_t row = (size_t)i * np;
  const float *W = L.W[j] + row, *Q = L.Q[j] + row;
  const float2 *P = L.X[j] + row, *T = L.T[j] + row;
  float accf = 0.0f;
  double acc = 0.0;
  for (int c = lane, t = 0; c < np; c += 32, ++t) {
    const float2 p = P[c], tt = T[c];
    accf += W[c] * (p.x + p.y) + Q[c] * (tt.x + tt.y);
    if ((t & 15) == 15) {
      acc += (double)accf;
      accf = 0.0f;
    }
  }
  acc += (double)accf;
  acc = warp_sum(acc);
  if (lane == 0) L.out[j][i] = 2.0 * (df_val(P[i]) - acc);
}

// out_i = (Y M)_ii = Mt_ii - sum_j W_ij Mt_ij  (Y = I - W, Mt = M^T), one warp per row
__global__ void row_dot_last_group_kernel(int np, DiagList L) {
  grid_wait();
  const int j = blockIdx.y;
  const int i = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= L.N[j]) return;
  const float* W = L.W[j];
  const float2* Mt = L.X[j];
  float accf = 0.0f;
  double acc = 0.0;
  for (int c = lane, t = 0; c < np; c += 32, ++t) {
    const float2 mm = Mt[(size_t)i * np + c];
    accf += W[(size_t)i * np + c] * (mm.x + mm.y);
    if ((t & 15) == 15) {
      acc += (double)accf;
      accf = 0.0f;
    }
  }
  acc += (double)accf;
  acc = warp_sum(acc);
  if (lane == 0) L.out[j][i] = df_val(Mt[(size_t)i * np + i]) - acc;
}

__global__ void get_diag_group_kernel(int np, DiagList L) {
  grid_wait();
  const int j = blockIdx.y;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < L.N[j]) L.out[j][i] = df_val(L.X[j][(size_t)i * np + i]);
}

// Epilogue options of one split product.  The side inputs of a symmetric product
// must be symmetric where out2 is written (E is read at the mirrored place too).
struct Epi {
  float alpha = 1.0f;
  const SplitMat* E = nullptr;
  float beta = 0.0f;
  const SplitMat* E2 = nullptr;
  float beta2 = 0.0f;
  const float2* E64 = nullptr;
  float beta64 = 0.0f;
  float diag = 0.0f;
  const double* dvec = nullptr;
  float dvec_scale = 1.0f;
  bool out64 = false;       // write C.d (and the operands of it) instead of C.f
  bool value = true;        // write the value of C
  bool convert = true;      // write the operands of C
  bool hi_only = false;     // only the hi operand (C enters single products only)
  SplitMat* V = nullptr;    // second result va C + vb E: value and operands
  float va = 0.0f, vb = 0.0f;
  int nseg = 3;             // 3: hi*hi + hi*lo + lo*hi; 1: hi*hi only
  int pairs = 1;            // 2: C = A B^T + B A^T, or A B^T + A2 B2^T with a second pair
};

// The recursion is carried in correction form so that its exact leading
// terms never pass through the rounded operands:
//   T_{k+1} = 2 T_k - 2 T_k W_k,  W_k = I - Y_k = I - (I + T_k^2)^-1,
// W_k from residual corrections written for W (Q = S - W - W S,
// W <- W + P - P W, P a polynomial in Q: plan.h), and the response chains as
//   M = 2 T1_k - A1 T_{k+1},  T1_{k+1} = M - W_k M.
// T_k, M and T1_k are FP64 values; W, S, Q, A1 FP32 values; every product
// operand is the hi/lo split of a value.
class EngineSplit : public Engine {
 public:
  explicit EngineSplit(int prec) : fmt_(operand_fmt(prec)) {}
  ~EngineSplit() override {
    for (auto& kv : tiles_) cudaFree(kv.second.first);
    if (err_) cudaFree(err_);
    free_e64();
    tc_group_cache_free(group_cache_);
  }

  // Symmetric-product tile lists for size np, uploaded on the stream that uses them (the
  // context's stream may be non-blocking, so a legacy-stream copy would not be ordered
  // before the first product).
  cudaError_t prep_tiles(int np, cudaStream_t s) {
    if (tiles_.count(np)) return cudaSuccess;
    const bool wide = (np % 256 == 0);
    std::vector<int> all, part;
    TcTiles t;
    size_t off[kTcWidths + 1];
    for (int w = 0; w < kTcWidths; ++w) {
      off[w] = all.size();
      if (tc_width(w) == 256 && !wide) continue;
      part = tc_sym_tiles(np, tc_width(w));
      t.nsym[w] = (int)part.size() / 2;
      all.insert(all.end(), part.begin(), part.end());
    }
    off[kTcWidths] = all.size();
    if (wide) {
      part = tc_sym_tiles_pair(np);
      t.npair = (int)part.size() / 2;
      all.insert(all.end(), part.begin(), part.end());
    }
    int* d = nullptr;
    RET(cudaMalloc((void**)&d, sizeof(int) * std::max<size_t>(all.size(), 2)));
    RET(cudaMemcpyAsync(d, all.data(), sizeof(int) * all.size(), cudaMemcpyHostToDevice, s));
    for (int w = 0; w < kTcWidths; ++w) t.sym[w] = d + off[w];
    t.pair = wide ? d + off[kTcWidths] : nullptr;
    tiles_[np] = {d, t};
    if (!err_) {
      RET(cudaMalloc((void**)&err_, sizeof(int)));
      RET(cudaMemsetAsync(err_, 0, sizeof(int), s));
    }
    return cudaStreamSynchronize(s);   // `all` is a host temporary
  }

  // the epilogue arguments of C = epi(A B^T)
  static void fill_args(TcArgs& a, int np, const SplitMat& A, const SplitMat& B, SplitMat& C, const Epi& e) {
    a.alpha = e.alpha;
    a.E = e.E ? e.E->f : nullptr;
    a.beta = e.beta;
    a.E2 = e.E2 ? e.E2->f : nullptr;
    a.beta2 = e.beta2;
    a.E64 = e.E64;
    a.beta64 = e.beta64;
    a.diag = e.diag;
    a.dvec = e.dvec;
    a.ndvec = e.dvec ? np : 0;
    a.dvec_scale = e.dvec_scale;
    a.out.f = (e.value && !e.out64) ? C.f : nullptr;
    a.out.d = e.out64 ? C.d : nullptr;
    if (e.convert) {
      a.out.hi = C.hi;
      a.out.lo = e.hi_only ? nullptr : C.lo;
      a.out.scale = C.scale;
    }
    if (e.V) {
      a.out2.f = e.V->f;
      a.out2.hi = e.V->hi;
      a.out2.lo = e.hi_only ? nullptr : e.V->lo;
      a.out2.scale = e.V->scale;
      a.va = e.va;
      a.vb = e.vb;
    }
    a.ldc = np;
    a.sa = A.scale;
    a.sb = B.scale;
  }

  void fill_shared(TcArgs& a, int np, const Epi& e, bool sym) const {
    a.nseg = e.nseg;
    a.pairs = e.pairs;
    a.sym = sym ? 1 : 0;
    a.fmt = fmt_;
    a.err = err_;
    // one-CTA-per-tile kernel, large products: the hi*hi sums split over both accumulators
    a.split_acc = (np >= kSplitAccMin) ? 1 : 0;
    a.chunk_kb = kChunkK / (fmt_ == 2 ? 32 : 64);
  }

  struct GemmOp {
    const SplitMat* A;
    const SplitMat* B;
    SplitMat* C;
    Epi e;
    double* stats;
    const SplitMat *A2 = nullptr, *B2 = nullptr;
  };

  void fill_problem(TcProblem& p, int np, const GemmOp& o) const {
    p.Ahi = o.A->hi;
    p.Alo = o.A->lo;
    p.Bhi = o.B->hi;
    p.Blo = o.B->lo;
    if (o.A2) {
      p.A2hi = o.A2->hi;
      p.A2lo = o.A2->lo;
      p.B2hi = o.B2->hi;
      p.B2lo = o.B2->lo;
    }
    fill_args(p.epi, np, *o.A, *o.B, *o.C, o.e);
  }

  cudaError_t gemm(cudaStream_t s, int np, const GemmOp& o, bool sym) {
    const Epi& e = o.e;
    double* stats = o.stats;
    RET(prep_tiles(np, s));
    const TcTiles& tl = tiles_[np].second;
    TcProblem p;
    fill_problem(p, np, o);
    fill_shared(p.epi, np, e, sym);
    RET(prof_begin(s));
    RET(gemm_tc(s, np, p, tl));
    // kind bits: 1 sym, 2 E, 4 E2, 8 E64, 16 second result, 32 double-float output
    const int kind = (sym ? 1 : 0) | (e.E ? 2 : 0) | (e.E2 ? 4 : 0) | (e.E64 ? 8 : 0) | (e.V ? 16 : 0) |
                     (e.out64 ? 32 : 0);
    RET(prof_end(s, 2.0 * (double)np * np * np * (sym ? 0.5 : 1.0) * e.pairs, kind));
    if (stats) stats[3] += (sym ? 0.5 : 1.0) * e.pairs;
    return cudaSuccess;
  }

  // ---- grouped operations (one launch over the systems of a lockstep group) ----

  static dim3 ew_grid(size_t count, int nsys) {
    return dim3((unsigned)std::max<size_t>(1, std::min<size_t>(nblk(count), kEwBlocks / nsys)), (unsigned)nsys);
  }

  // One product per op, all in one grouped launch (ops share sym, nseg, pairs).
  cudaError_t gemm_group(cudaStream_t s, int np, std::vector<GemmOp>& ops, bool sym) {
    if (ops.empty()) return cudaSuccess;
    if (ops.size() == 1) return gemm(s, np, ops[0], sym);
    RET(prep_tiles(np, s));
    const TcTiles& tl = tiles_[np].second;
    const Epi& e0 = ops[0].e;
    TcArgs shared;
    fill_shared(shared, np, e0, sym);
    std::vector<TcProblem> probs(ops.size());
    for (size_t i = 0; i < ops.size(); ++i) {
      const GemmOp& o = ops[i];
      fill_problem(probs[i], np, o);
      if (o.stats) o.stats[3] += (sym ? 0.5 : 1.0) * e0.pairs;
    }
    if (!group_cache_) group_cache_ = tc_group_cache_new();
    RET(prof_begin(s));
    RET(gemm_tc_group(s, np, probs.data(), (int)probs.size(), shared, tl, group_cache_));
    const int kind = 64 | (sym ? 1 : 0) | (e0.E ? 2 : 0) | (e0.E2 ? 4 : 0) | (e0.E64 ? 8 : 0) | (e0.V ? 16 : 0) |
                     (e0.out64 ? 32 : 0);
    return prof_end(s, (double)ops.size() * 2.0 * (double)np * np * np * (sym ? 0.5 : 1.0) * e0.pairs, kind);
  }

  cudaError_t foe(cudaStream_t s, MatSet& m, const double* H, int N, double mu, double sc,
                  const std::vector<LevelPlan>& plan, double* stats, const double* dpar) override {
    std::vector<FoeJob> jobs(1);
    jobs[0].m = &m;
    jobs[0].H = H;
    jobs[0].N = N;
    jobs[0].mu = mu;
    jobs[0].plan = &plan;
    jobs[0].stats = stats;
    jobs[0].dpar = dpar;
    return foe_group(s, jobs, sc);
  }

  // Linear combination of matrices per system into Y[i] and its operands.
  cudaError_t combine_group(cudaStream_t s, int np, CombList& L, const std::vector<SplitMat*>& Y, bool hi_only) {
    L.n = (int)Y.size();
    for (int i = 0; i < L.n; ++i) {
      L.Y[i] = Y[i]->f;
      L.hi[i] = Y[i]->hi;
      L.lo[i] = hi_only ? nullptr : Y[i]->lo;
      L.scale[i] = Y[i]->scale;
    }
    RET(launch_chained(s, ew_grid((size_t)np * np / 4, L.n), 256, 0, combine_group_kernel, np, fmt_, L));
    return cudaSuccess;
  }

  // operands of a matrix from its value, in place
  cudaError_t operands(cudaStream_t s, SplitMat& m, int np) {
    CombList L;
    L.X[0][0] = m.f;
    L.X[1][0] = L.X[2][0] = nullptr;
    L.g[0][0] = L.g[2][0] = L.g[3][0] = 0.f;
    L.g[1][0] = 1.f;
    L.dg[0] = nullptr;
    const std::vector<SplitMat*> Y(1, &m);
    return combine_group(s, np, L, Y, false);
  }

  // The chains' matrices serve as scratch of the expansion and of dT_n/dmu, at the unit scale.
  static void unit_scales(MatSet& m) {
    for (SplitMat* x : {&m.sA1, &m.sMt, &m.sT1a, &m.sT1b, &m.sYw}) x->scale = m.scales;
  }

  // The recursion of every job's system in lockstep: each product of a level is one grouped
  // launch over the jobs that need it (a job runs its own plan).
  cudaError_t foe_group(cudaStream_t s, std::vector<FoeJob>& jobs, double sc) override {
    const int B = (int)jobs.size();
    if (B == 0) return cudaSuccess;
    if (B > kMaxGroup) {
      for (int i = 0; i < B; i += kMaxGroup) {
        std::vector<FoeJob> part(jobs.begin() + i, jobs.begin() + std::min(B, i + kMaxGroup));
        RET(foe_group(s, part, sc));
      }
      return cudaSuccess;
    }
    const int np = jobs[0].m->np, n = jobs[0].m->n;
    for (auto& j : jobs)
      if (j.m->np != np || j.m->n != n) return cudaErrorInvalidValue;
    const size_t cnt = (size_t)np * np;
    T0List tl;
    tl.n = B;
    for (int i = 0; i < B; ++i) {
      FoeJob& j = jobs[i];
      MatSet& m = *j.m;
      unit_scales(m);
      tl.N[i] = j.N;
      tl.H[i] = j.H;
      tl.mu[i] = j.mu;
      tl.t0[i] = m.t0max;
      tl.dpar[i] = j.dpar;
      tl.T0[i] = m.sT[0].d;
      tl.hi[i] = m.sT[0].hi;
      tl.lo[i] = m.sT[0].lo;
      tl.scales[i] = m.scales;
      tl.t0_dev[i] = m.t0_dev;
    }
    RET(launch_chained(s, ew_grid(cnt / 4, B), 256, 0, t0_init_group_kernel, np, n, fmt_, kPassT0, sc, tl));
    std::vector<SplitMat*> W(B), Wn(B);
    // scratch of the corrections: matrices of the response chains, which are free here
    auto Sk = [](MatSet& m, int k) -> SplitMat* { return (k & 1) ? &m.sT1b : &m.sS; };   // S_k beside S_{k-1}
    for (int k = 0; k < n; ++k) {
      std::vector<GemmOp> ops;
      for (auto& j : jobs) ops.push_back({&j.m->sT[k], &j.m->sT[k], Sk(*j.m, k), Epi(), j.stats});   // S = T^2
      RET(gemm_group(s, np, ops, true));
      // the iterates alternate between sY[k] and the work matrix; the start is chosen by the
      // parity of the rounds so that W_k always ends in sY[k] (the buffers every later use, and
      // a captured graph of this pass, refer to)
      CombList cl;
      int rounds = 0;
      for (int i = 0; i < B; ++i) {
        FoeJob& j = jobs[i];
        MatSet& m = *j.m;
        const LevelPlan& p = (*j.plan)[k];
        rounds = std::max(rounds, p.inv.n);
        W[i] = (p.inv.n % 2 == 1) ? &m.sYw : &m.sY[k];
        Wn[i] = (W[i] == &m.sY[k]) ? &m.sYw : &m.sY[k];
        cl.X[0][i] = k > 0 ? m.sY[k - 1].f : nullptr;                            // W0 (plan.h)
        cl.X[1][i] = p.nb > 2 ? Sk(m, k)->f : nullptr;
        cl.X[2][i] = p.nb > 3 ? Sk(m, k - 1)->f : nullptr;
        for (int q = 0; q < 4; ++q) cl.g[q][i] = (float)p.g[q];
        cl.dg[i] = j.dpar ? j.dpar + 1 + 4 * k : nullptr;
      }
      RET(combine_group(s, np, cl, W, false));
      for (int r = 0; r < rounds; ++r) {
        // Q = S - W - W S and P = Q - Q^2 + ..: functions of one matrix, so every product is symmetric
        std::vector<GemmOp> oq, o2, o3, o5, ow;
        for (int i = 0; i < B; ++i) {
          FoeJob& j = jobs[i];
          const InvOrders& inv = (*j.plan)[k].inv;
          if (r >= inv.n) continue;
          MatSet& m = *j.m;
          const int order = inv.order[r];
          SplitMat* P = &m.sQ;
          Epi eq;
          eq.alpha = -1.f;
          eq.E = Sk(m, k);
          eq.beta = 1.f;
          eq.E2 = W[i];
          eq.beta2 = -1.f;
          oq.push_back({W[i], Sk(m, k), &m.sQ, eq, j.stats});
          Epi e2;
          e2.E = &m.sQ;
          if (order == 3) {                                                      // P = Q - Q^2
            e2.alpha = -1.f;
            e2.beta = 1.f;
            o3.push_back({&m.sQ, &m.sQ, &m.sA1, e2, j.stats});
            P = &m.sA1;
          }
          if (order == 5) {                                                      // P = V + V Q^2, V = Q - Q^2
            e2.value = false;
            e2.V = &m.sMt;
            e2.va = -1.f;
            e2.vb = 1.f;
            o2.push_back({&m.sQ, &m.sQ, &m.sA1, e2, j.stats});
            Epi e5;
            e5.E = &m.sMt;
            e5.beta = 1.f;
            o5.push_back({&m.sMt, &m.sA1, &m.sT1a, e5, j.stats});
            P = &m.sT1a;
          }
          Epi ew;                                                                // W <- W + P - P W
          ew.alpha = -1.f;
          ew.E = W[i];
          ew.beta = 1.f;
          ew.E2 = P;
          ew.beta2 = 1.f;
          ow.push_back({P, W[i], Wn[i], ew, j.stats});
          std::swap(W[i], Wn[i]);
          if (j.stats) j.stats[1] += 1;
        }
        RET(gemm_group(s, np, oq, true));
        RET(gemm_group(s, np, o3, true));
        RET(gemm_group(s, np, o2, true));
        RET(gemm_group(s, np, o5, true));
        RET(gemm_group(s, np, ow, true));
      }
      std::vector<GemmOp> ot;
      for (auto& j : jobs) {
        MatSet& m = *j.m;
        Epi et;                                                                   // T' = 2T - 2 T W
        et.alpha = -2.f;
        et.E64 = m.sT[k].d;
        et.beta64 = 2.0f;
        et.out64 = true;
        ot.push_back({&m.sT[k], &m.sY[k], &m.sT[k + 1], et, j.stats});
      }
      RET(gemm_group(s, np, ot, true));
    }
    return cudaSuccess;
  }

  cudaError_t mu_derivative(cudaStream_t s, MuJob& j, double amp) override {
    std::vector<MuJob> jobs(1, j);
    return mu_derivative_group(s, jobs, amp);
  }

  cudaError_t mu_derivative_group(cudaStream_t s, std::vector<MuJob>& jobs, double amp) override {
    const int B = (int)jobs.size();
    if (B == 0) return cudaSuccess;
    if (B > kMaxGroup) {
      for (int i = 0; i < B; i += kMaxGroup) {
        std::vector<MuJob> part(jobs.begin() + i, jobs.begin() + std::min(B, i + kMaxGroup));
        RET(mu_derivative_group(s, part, amp));
      }
      return cudaSuccess;
    }
    const int np = jobs[0].m->np, n = jobs[0].m->n;
    for (auto& j : jobs)
      if (j.m->np != np || j.m->n != n) return cudaErrorInvalidValue;
    const bool single = (mu_nseg_ == 1);
    Epi base;
    base.nseg = mu_nseg_;
    base.hi_only = single;
    // the matrices of the response chains and of the expansion's corrections are idle here
    std::vector<GemmOp> o1;
    for (auto& j : jobs) {
      unit_scales(*j.m);
      o1.push_back({&j.m->sT[0], &j.m->sT[0], &j.m->sS, base, j.stats});
    }
    RET(gemm_group(s, np, o1, true));
    std::vector<SplitMat*> Z(B), Zn(B), C(B);
    CombList cz;
    int rounds = 0;
    for (int i = 0; i < B; ++i) {
      MuJob& j = jobs[i];
      const ResolventPlan& p = *j.plan;
      rounds = std::max(rounds, p.inv.n);
      Z[i] = &j.m->sYw;
      Zn[i] = &j.m->sT1b;
      Z[i]->scale = Zn[i]->scale = j.m->scales + 2 + n;
      cz.X[0][i] = j.m->sS.f;
      cz.X[1][i] = cz.X[2][i] = nullptr;
      cz.g[0][i] = (float)p.z0;
      cz.g[1][i] = (float)p.z1;
      cz.g[2][i] = cz.g[3][i] = 0.f;
      cz.dg[i] = j.dpar;
    }
    RET(combine_group(s, np, cz, Z, single));
    for (int r = 0; r < rounds; ++r) {
      std::vector<GemmOp> oq, o2, o3, o5, ow;
      for (int i = 0; i < B; ++i) {
        MuJob& j = jobs[i];
        if (r >= j.plan->inv.n) continue;
        MatSet& m = *j.m;
        const int order = j.plan->inv.order[r];
        SplitMat* P = &m.sQ;
        Epi eq = base;                                                            // R = I - Z + S Z
        eq.E = Z[i];
        eq.beta = -1.f;
        eq.diag = 1.f;
        oq.push_back({&m.sS, Z[i], &m.sQ, eq, j.stats});
        Epi e2 = base;
        e2.E = &m.sQ;
        if (order == 3) {                                                         // P = R + R^2
          e2.beta = 1.f;
          o3.push_back({&m.sQ, &m.sQ, &m.sA1, e2, j.stats});
          P = &m.sA1;
        }
        if (order == 5) {                                                         // P = V + V R^2, V = R + R^2
          e2.value = false;
          e2.V = &m.sMt;
          e2.va = 1.f;
          e2.vb = 1.f;
          o2.push_back({&m.sQ, &m.sQ, &m.sA1, e2, j.stats});
          Epi e5 = base;
          e5.E = &m.sMt;
          e5.beta = 1.f;
          o5.push_back({&m.sMt, &m.sA1, &m.sT1a, e5, j.stats});
          P = &m.sT1a;
        }
        Epi ew = base;                                                            // Z <- Z + P Z
        ew.E = Z[i];
        ew.beta = 1.f;
        ow.push_back({P, Z[i], Zn[i], ew, j.stats});
        std::swap(Z[i], Zn[i]);
      }
      RET(gemm_group(s, np, oq, true));
      RET(gemm_group(s, np, o3, true));
      RET(gemm_group(s, np, o2, true));
      RET(gemm_group(s, np, o5, true));
      RET(gemm_group(s, np, ow, true));
    }
    CombList cc;
    std::vector<GemmOp> oc, ot;
    DiagList dl;
    dl.n = B;
    int maxN = 0;
    for (int i = 0; i < B; ++i) {
      MuJob& j = jobs[i];
      MatSet& m = *j.m;
      C[i] = &m.sMt;
      cc.X[0][i] = m.sY[n - 1].f;                                                 // C = I - 2 W_{n-1}
      cc.X[1][i] = cc.X[2][i] = nullptr;
      cc.g[0][i] = 1.f;
      cc.g[1][i] = -2.f;
      cc.g[2][i] = cc.g[3][i] = 0.f;
      cc.dg[i] = nullptr;
      oc.push_back({&m.sMt, &m.sMt, &m.sA1, base, j.stats});
      Epi et = base;
      et.alpha = (float)amp;
      et.out64 = true;
      et.convert = false;
      ot.push_back({&m.sA1, Z[i], &m.sTmu, et, j.stats});
      dl.N[i] = j.N;
      dl.X[i] = m.sTmu.d;
      dl.out[i] = j.out_diag;
      maxN = std::max(maxN, j.N);
    }
    RET(combine_group(s, np, cc, C, single));
    RET(gemm_group(s, np, oc, true));
    RET(gemm_group(s, np, ot, true));
    RET(launch_chained(s, dim3((maxN + 255) / 256, B), 256, 0, get_diag_group_kernel, np, dl));
    return cudaSuccess;
  }

  cudaError_t chain(cudaStream_t s, MatSet& m, const double* dvec, int N, double* out_diag,
                    double* stats) override {
    std::vector<ChainJob> jobs(1);
    jobs[0].m = &m;
    jobs[0].dvec = dvec;
    jobs[0].N = N;
    jobs[0].out_diag = out_diag;
    jobs[0].stats = stats;
    return chain_group(s, jobs);
  }

  // A level of a chain in two launches instead of three: with Y T = T' / 2 and T T' = 2 W,
  //   T1' = 2 Y (T1 - T T1 T) Y = 2 P - 2 (P W + Q T'),  P = Y T1 = T1 - W T1,  Q = T' T1 / 4,
  // P and Q side by side, then one symmetric product over two K pairs.  A level is 3 n^3 multiply-adds this
  // way and 2.5 n^3 in three launches, so it is taken where launches count: up to 128 tiles of 128 x 128 per
  // matrix of the probes side by side, less than one for each SM.  The systems of a lockstep group do not
  // count: each gives the bits of its own run.  Three and two launches, us: response at n = 1024 669 and
  // 612, two steps of 24 atoms 2305 and 2102, of 8 systems of 57 atoms 4439 and 4379, 150 atoms (n = 640)
  // 2104 and 2002, 333 atoms TF32x3 (1408, 121 tiles) 5771 and 5594; 512 atoms (2048, 256 tiles) 7116 and
  // 7270, 48 probes at n = 384 3577 and 3703.
  static bool two_step(int np, int side) { return (long long)side * (np / 128) * (np / 128) <= 128; }

  cudaError_t chain_two_step(cudaStream_t s, std::vector<ChainJob>& jobs, int np, int n) {
    const int B = (int)jobs.size(), nseg = probe_nseg_;
    const bool single = (nseg == 1);
    const size_t cnt = (size_t)np * np;
    for (int k = 0; k < n; ++k) {
      const bool last = (k == n - 1);
      P0List pl;
      pl.n = B;
      std::vector<GemmOp> op, ot;
      for (int i = 0; i < B; ++i) {
        MatSet& m = *jobs[i].m;
        const float* cs = m.chain_scales + 3 * k;
        SplitMat *Q = &m.sA1, *P = &m.sMt, *T1 = (k & 1) ? &m.sT1b : &m.sT1a, *T1n = (k & 1) ? &m.sT1a : &m.sT1b;
        Q->scale = cs;
        P->scale = cs + 1;
        T1n->scale = cs + 2;
        if (k == 0) {
          pl.W[i] = m.sY[0].f;
          pl.T[i] = m.sT[1].d;
          pl.d[i] = jobs[i].dvec;
          pl.Pf[i] = single && !last ? P->f : nullptr;
          pl.Pd[i] = P->d;
          pl.Qf[i] = Q->f;
          pl.Phi[i] = P->hi;
          pl.Plo[i] = single ? nullptr : P->lo;
          pl.Qhi[i] = Q->hi;
          pl.Qlo[i] = single ? nullptr : Q->lo;
          pl.Ps[i] = P->scale;
          pl.Qs[i] = Q->scale;
        } else {
          Epi ep;                                                                // P = T1 - W T1
          ep.alpha = -1.f;
          if (single) {
            ep.E = T1;
            ep.beta = 1.f;
          } else {
            ep.E64 = T1->d;
            ep.beta64 = 1.f;
          }
          ep.out64 = !single || last;
          ep.convert = !last;                                                    // the last ones are only reduced
          ep.hi_only = single;
          ep.nseg = nseg;
          op.push_back({&m.sY[k], T1, P, ep, jobs[i].stats});
          Epi eq;                                                                // Q = T' T1 / 4
          eq.alpha = 0.25f;
          eq.value = last;
          eq.convert = !last;
          eq.hi_only = single;
          eq.nseg = nseg;
          op.push_back({&m.sT[k + 1], T1, Q, eq, jobs[i].stats});
        }
        Epi et;                                                                  // T1' = 2 P - 2 (P W + Q T')
        et.alpha = -2.f;
        if (single) {
          et.E = P;
          et.beta = 2.f;
          et.hi_only = true;
        } else {
          et.E64 = P->d;
          et.beta64 = 2.f;
          et.out64 = true;
        }
        et.nseg = nseg;
        et.pairs = 2;
        ot.push_back({P, &m.sY[k], T1n, et, jobs[i].stats, Q, &m.sT[k + 1]});
      }
      if (k == 0)
        RET(launch_chained(s, ew_grid(cnt / 4, B), 256, 0, level0_P_group_kernel, np, fmt_, pl));
      else
        RET(gemm_group(s, np, op, false));
      if (!last) {
        RET(gemm_group(s, np, ot, true));
        continue;
      }
      DiagList dl;
      dl.n = B;
      int maxN = 0;
      for (int i = 0; i < B; ++i) {
        MatSet& m = *jobs[i].m;
        dl.N[i] = jobs[i].N;
        dl.W[i] = m.sY[k].f;
        dl.X[i] = m.sMt.d;
        dl.Q[i] = m.sA1.f;
        dl.T[i] = m.sT[k + 1].d;
        dl.out[i] = jobs[i].out_diag;
        maxN = std::max(maxN, jobs[i].N);
      }
      RET(launch_chained(s, dim3((maxN + 7) / 8, B), 256, 0, row_dot_two_group_kernel, np, dl));
    }
    return cudaSuccess;
  }

  // Response chains of several systems (or several probes of one system, each with its own
  // chain matrices) in lockstep, every product a grouped launch.
  cudaError_t chain_group(cudaStream_t s, std::vector<ChainJob>& jobs) override {
    const int B = (int)jobs.size();
    if (B == 0) return cudaSuccess;
    if (B > kMaxGroup) {
      for (int i = 0; i < B; i += kMaxGroup) {
        std::vector<ChainJob> part(jobs.begin() + i, jobs.begin() + std::min(B, i + kMaxGroup));
        RET(chain_group(s, part));
      }
      return cudaSuccess;
    }
    const int np = jobs[0].m->np, n = jobs[0].m->n;
    for (auto& j : jobs)
      if (j.m->np != np || j.m->n != n) return cudaErrorInvalidValue;
    const size_t cnt = (size_t)np * np;
    const int nseg = probe_nseg_;
    // A single-product chain keeps M and T1 as FP32 values with hi operands only: its products
    // carry ~2^-11 relative error, so the double-float values and lo operands of the three-product
    // chain would add traffic and no accuracy.  The last level still writes the double-float array
    // the reductions read (with a zero low word).
    const bool single = (nseg == 1);
    const bool two = two_step(np, jobs[0].side);
    ChainScaleList sl;
    sl.n = B;
    for (int i = 0; i < B; ++i) {
      sl.ts[i] = two ? jobs[i].m->scales + 1 : nullptr;
      sl.d[i] = jobs[i].dvec;
      sl.t0[i] = jobs[i].m->t0_dev;
      sl.scales[i] = jobs[i].m->chain_scales;
    }
    RET(launch_chained(s, B, 256, 0, chain_scales_kernel, np, n, sl));
    std::vector<SplitMat*> T1(B), T1n(B), A1s(B), Mts(B);
    for (int i = 0; i < B; ++i) {
      T1[i] = &jobs[i].m->sT1a;
      T1n[i] = &jobs[i].m->sT1b;
      A1s[i] = &jobs[i].m->sA1;
      Mts[i] = &jobs[i].m->sMt;
    }
    if (two) return chain_two_step(s, jobs, np, n);
    for (int k = 0; k < n; ++k) {
      const bool last = (k == n - 1);
      for (int i = 0; i < B; ++i) {
        const float* cs = jobs[i].m->chain_scales + 3 * k;
        A1s[i]->scale = cs;
        Mts[i]->scale = cs + 1;
        T1n[i]->scale = cs + 2;
      }
      Epi em;                                                                    // Mt = 2 T1 - T_{k+1} A1
      em.alpha = -1.f;
      em.out64 = !single || last;
      em.hi_only = single;
      em.convert = !last;                                                        // the last M is only reduced
      em.nseg = nseg;
      std::vector<GemmOp> om;
      if (k == 0) {
        A1List al;
        al.n = B;
        for (int i = 0; i < B; ++i) {
          al.T0[i] = jobs[i].m->sT[0].d;
          al.d[i] = jobs[i].dvec;
          al.hi[i] = A1s[i]->hi;
          al.lo[i] = single ? nullptr : A1s[i]->lo;
          al.scale[i] = A1s[i]->scale;
        }
        RET(launch_chained(s, ew_grid(cnt / 4, B), 256, 0, level0_A1_group_kernel, np, fmt_, al));
        for (int i = 0; i < B; ++i) {
          Epi e = em;
          e.dvec = jobs[i].dvec;
          e.dvec_scale = 2.f;
          om.push_back({&jobs[i].m->sT[k + 1], A1s[i], Mts[i], e, jobs[i].stats});
        }
      } else {
        // A1 = T T1 + T1 T (T, T1 symmetric): one symmetric-output product over the two K pairs; only
        // its operands are needed
        std::vector<GemmOp> oa;
        for (int i = 0; i < B; ++i) {
          Epi ea;
          ea.value = false;
          ea.hi_only = single;
          ea.nseg = nseg;
          ea.pairs = 2;
          oa.push_back({&jobs[i].m->sT[k], T1[i], A1s[i], ea, jobs[i].stats});
        }
        RET(gemm_group(s, np, oa, true));
        for (int i = 0; i < B; ++i) {
          Epi e = em;
          if (single) {
            e.E = T1[i];                                                          // FP32
            e.beta = 2.0f;
          } else {
            e.E64 = T1[i]->d;
            e.beta64 = 2.0f;
          }
          om.push_back({&jobs[i].m->sT[k + 1], A1s[i], Mts[i], e, jobs[i].stats});
        }
      }
      RET(gemm_group(s, np, om, false));
      if (last) {
        DiagList dl;
        dl.n = B;
        int maxN = 0;
        for (int i = 0; i < B; ++i) {
          dl.N[i] = jobs[i].N;
          dl.W[i] = jobs[i].m->sY[k].f;
          dl.X[i] = Mts[i]->d;
          dl.out[i] = jobs[i].out_diag;
          maxN = std::max(maxN, jobs[i].N);
        }
        RET(launch_chained(s, dim3((maxN + 7) / 8, B), 256, 0, row_dot_last_group_kernel, np, dl));
        return cudaSuccess;
      }
      std::vector<GemmOp> oy;
      for (int i = 0; i < B; ++i) {
        Epi ey;                                                                  // T1' = Mt - Mt W
        ey.alpha = -1.f;                                                         // (symmetric: = M - W M)
        if (single) {
          ey.E = Mts[i];
          ey.beta = 1.0f;
          ey.hi_only = true;
        } else {
          ey.E64 = Mts[i]->d;
          ey.beta64 = 1.0f;
          ey.out64 = true;
        }
        ey.nseg = nseg;
        oy.push_back({Mts[i], &jobs[i].m->sY[k], T1n[i], ey, jobs[i].stats});
      }
      RET(gemm_group(s, np, oy, true));
      std::swap(T1, T1n);
    }
    return cudaSuccess;
  }

  const int* device_error() const override { return err_; }
  void set_chain_segments(int probe_nseg, int mu_nseg) override {
    probe_nseg_ = (probe_nseg == 1) ? 1 : 3;
    mu_nseg_ = (mu_nseg == 1) ? 1 : 3;
  }

  cudaError_t trace_tn(cudaStream_t s, MatSet& m, int N, double* out) override {
    diag_sum_d_kernel<<<1, 1024, 0, s>>>(N, m.np, m.sT[m.n].d, out);
    note_launch();
    return cudaGetLastError();
  }

  cudaError_t density_out(cudaStream_t s, MatSet& m, int N, double dmu, const double*, double* ddiag,
                          double* D) override {
    density_out_d_kernel<<<nblk((size_t)m.np * m.np), 256, 0, s>>>(N, m.np, m.sT[m.n].d, m.sTmu.d, dmu, ddiag, D);
    note_launch();
    return cudaGetLastError();
  }

  cudaError_t entropy(cudaStream_t s, MatSet& m, int N, double, int n_sq, double, double, const double* D,
                      const double*, double* work, double* out) override {
    // FP64 route from the split values: T_0 from its double-float value, Y_k = I - W_k
    const size_t cnt = (size_t)m.np * m.np;
    if (cnt > e64_count_) {
      free_e64();
      for (double*& p : e64_) {
        const cudaError_t e = cudaMalloc((void**)&p, cnt * sizeof(double));
        if (e != cudaSuccess) {
          p = nullptr;
          free_e64();
          return e;
        }
      }
      e64_count_ = cnt;
    }
    double* T0 = e64_[5];
    df_to_f64_kernel<<<nblk(cnt), 256, 0, s>>>(cnt, m.sT[0].d, T0);
    note_launch();
    RET(cudaGetLastError());
    auto load_Y = [&](int k, double* dst) -> cudaError_t {
      ident_minus_f32_to_f64_kernel<<<nblk(cnt), 256, 0, s>>>(cnt, N, m.np, m.sY[k].f, dst);
      note_launch();
      return cudaGetLastError();
    };
    // artanh series: terms until 2^(n+1) t0max^(2j+1) / (2j+1) N < 1e-10
    int nterms = 1;
    const double t = m.t0max;
    while (nterms < 6 && std::ldexp(1.0, n_sq + 1) * std::pow(t, 2 * nterms + 1) / (2 * nterms + 1) * N > 1e-10)
      ++nterms;
    return entropy_fp64(s, N, m.np, m.n, n_sq, T0, load_Y, ent_, e64_[0], e64_[1], e64_[2], e64_[3],
                        e64_[4], nterms, D, work, out);
  }

  int* err_ = nullptr;

 private:
  void free_e64() {
    for (double*& p : e64_) {
      if (p) cudaFree(p);
      p = nullptr;
    }
    e64_count_ = 0;
  }

  double* e64_[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};   // FP64 matrices of the entropy (first use)
  size_t e64_count_ = 0;                                                      // elements of each: the largest system's
  int fmt_;   // operand format: 0 FP16, 1 BF16, 2 TF32
  int probe_nseg_ = 3;
  int mu_nseg_ = 3;
  std::unordered_map<int, std::pair<int*, TcTiles>> tiles_;
  TcGroupCache* group_cache_ = nullptr;
};

// which value arrays a matrix keeps
enum { kF = 1, kD = 2 };

// Zeroing runs on the stream `s` that later uses the matrix.
// esz: bytes of one operand element (2: FP16/BF16, 4: TF32)
cudaError_t alloc_split(SplitMat& m, int np, int esz, const float* scale, int what, cudaStream_t s) {
  const size_t cnt = (size_t)np * np;
  if (what & kF) {
    RET(cudaMalloc((void**)&m.f, cnt * sizeof(float)));
    RET(cudaMemsetAsync(m.f, 0, cnt * sizeof(float), s));
  }
  if (what & kD) {
    RET(cudaMalloc((void**)&m.d, cnt * sizeof(float2)));
    RET(cudaMemsetAsync(m.d, 0, cnt * sizeof(float2), s));
  }
  RET(cudaMalloc((void**)&m.hi, cnt * esz));
  RET(cudaMalloc((void**)&m.lo, cnt * esz));
  RET(cudaMemsetAsync(m.hi, 0, cnt * esz, s));
  RET(cudaMemsetAsync(m.lo, 0, cnt * esz, s));
  m.scale = scale;
  return cudaSuccess;
}

void free_split(SplitMat& m) {
  if (m.f) cudaFree(m.f);
  if (m.d) cudaFree(m.d);
  if (m.hi) {
    tc_forget_maps(m.hi);
    cudaFree(m.hi);
  }
  if (m.lo) {
    tc_forget_maps(m.lo);
    cudaFree(m.lo);
  }
  m.f = nullptr;
  m.d = nullptr;
  m.hi = m.lo = nullptr;
}

}  // namespace

Engine* make_split_engine(int prec) {
  if (!is_split_prec(prec)) return nullptr;
  return new EngineSplit(prec);
}

cudaError_t alloc_matset_split(MatSet& m, cudaStream_t s) {
  const int np = m.np, n = m.n, esz = operand_bytes(m.prec);
  const size_t nscale = 3 + (size_t)n + 3 * (size_t)n + 1;
  RET(cudaMalloc((void**)&m.scales, sizeof(float) * nscale));
  std::vector<float> init(nscale, kUnitScale);
  RET(cudaMemcpyAsync(m.scales, init.data(), sizeof(float) * nscale, cudaMemcpyHostToDevice, s));
  RET(cudaStreamSynchronize(s));   // init is a host temporary
  m.chain_scales = m.scales + 3 + n;
  m.t0_dev = m.chain_scales + 3 * n;
  m.sT.assign(n + 1, SplitMat());
  m.sY.assign(n, SplitMat());
  for (int k = 0; k <= n; ++k) RET(alloc_split(m.sT[k], np, esz, m.scales + 1 + k, kD, s));
  for (auto& x : m.sY) RET(alloc_split(x, np, esz, m.scales, kF, s));
  struct W {
    SplitMat* m;
    int what;
  } w[] = {{&m.sS, kF},  {&m.sQ, kF},  {&m.sYw, kF},  {&m.sA1, kF},
           {&m.sMt, kD | kF}, {&m.sT1a, kD | kF}, {&m.sT1b, kD | kF}, {&m.sTmu, kD}};
  for (auto& x : w) RET(alloc_split(*x.m, np, esz, m.scales, x.what, s));
  return cudaSuccess;
}

// A chain slot: a view of a system's expansion matrices (T_k, W_k shared) with its own
// response-chain matrices (A1, M, T1 twice) and their scalars, so that several probes of
// one system can run their chains side by side (grouped launches).  After a failure free_chain_slot
// gives back what the slot got: nothing of the base's is left in what it frees.
cudaError_t alloc_chain_slot(MatSet& slot, const MatSet& base, cudaStream_t s) {
  slot = base;
  const int np = base.np, esz = operand_bytes(base.prec);
  slot.chain_scales = nullptr;
  for (SplitMat* x : {&slot.sA1, &slot.sMt, &slot.sT1a, &slot.sT1b, &slot.sTmu}) *x = SplitMat();
  RET(cudaMalloc((void**)&slot.chain_scales, sizeof(float) * 3 * (size_t)base.n));
  RET(alloc_split(slot.sA1, np, esz, base.scales, kF, s));
  RET(alloc_split(slot.sMt, np, esz, base.scales, kD | kF, s));
  RET(alloc_split(slot.sT1a, np, esz, base.scales, kD | kF, s));
  RET(alloc_split(slot.sT1b, np, esz, base.scales, kD | kF, s));
  return cudaSuccess;
}

void free_chain_slot(MatSet& slot) {
  SplitMat* w[] = {&slot.sA1, &slot.sMt, &slot.sT1a, &slot.sT1b};
  for (SplitMat* x : w) free_split(*x);
  if (slot.chain_scales) cudaFree(slot.chain_scales);
  slot.chain_scales = nullptr;
  slot.sT.clear();
  slot.sY.clear();
}

// bytes of one chain slot of size np
size_t chain_slot_bytes(int np, int prec) {
  return (size_t)np * np * (8 + 3 * 16 + 4 * 2 * (operand_bytes(prec) - 2));
}

void free_matset_split(MatSet& m) {
  for (auto& x : m.sT) free_split(x);
  for (auto& x : m.sY) free_split(x);
  m.sT.clear();
  m.sY.clear();
  SplitMat* w[] = {&m.sS, &m.sQ, &m.sYw, &m.sA1, &m.sMt, &m.sT1a, &m.sT1b, &m.sTmu};
  for (SplitMat* x : w) free_split(*x);
  if (m.scales) cudaFree(m.scales);
  m.scales = m.chain_scales = m.t0_dev = nullptr;
}

// ---- self-test of the tensor-core product against the FP64 product ----

namespace {

__global__ void fill_random_kernel(size_t count, int np, uint64_t seed, int sym, double* out) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= count) return;
  size_t i = idx / np, j = idx % np;
  if (sym && j < i) {
    const size_t t = i;
    i = j;
    j = t;
  }
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (i * (uint64_t)np + j + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  out[idx] = ((double)(z >> 11) * (1.0 / 9007199254740992.0)) * 2.0 - 1.0;
}

__global__ void to_f32_kernel(size_t count, const double* __restrict__ x, float* __restrict__ f) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx < count) f[idx] = (float)x[idx];
}

__global__ void diff_f32_kernel(size_t count, const float* __restrict__ a, const float* __restrict__ b,
                                double* __restrict__ out) {
  __shared__ double sh[32];
  double m = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs((double)a[i] - (double)b[i]));
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, sh[w]);
    atomicMax(reinterpret_cast<unsigned long long*>(out), (unsigned long long)__double_as_longlong(t));
  }
}

__global__ void max_abs_diff_kernel(size_t count, const float* __restrict__ a, const double* __restrict__ b,
                                    double* __restrict__ out) {
  __shared__ double sh[32];
  double m = 0.0;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x)
    m = fmax(m, fabs((double)a[i] - b[i]));
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = fmax(t, sh[w]);
    unsigned long long* o = reinterpret_cast<unsigned long long*>(out);
    atomicMax(o, (unsigned long long)__double_as_longlong(t));
  }
}

}  // namespace

// Timing of the plain-FP64 product (the product of the FP64 path) at size n: one warm-up
// product at 128, then one timed product at n (sym: symmetric-output mode, half the tiles).
// Writes [0, 0, 0, ms per product].
int selftest_gemm_f64(int n, int sym, double* result) {
  const size_t cnt = (size_t)n * n;
  double *A = nullptr, *B = nullptr, *C = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  float ms = 0.f;
  int rc = -2;
  EpiF64 e;
  if (cudaMalloc((void**)&A, cnt * 8) || cudaMalloc((void**)&B, cnt * 8) || cudaMalloc((void**)&C, cnt * 8))
    goto done;
  fill_random_kernel<<<nblk(cnt), 256>>>(cnt, n, 11, 0, A);
  note_launch();
  fill_random_kernel<<<nblk(cnt), 256>>>(cnt, n, 23, sym, B);
  note_launch();
  if (gemm_f64_nt(nullptr, 128, 128, 128, A, n, B, n, C, n, e, sym != 0)) goto done;
  if (cudaEventCreate(&e0) || cudaEventCreate(&e1)) goto done;
  cudaEventRecord(e0, nullptr);
  if (gemm_f64_nt(nullptr, n, n, n, A, n, B, n, C, n, e, sym != 0)) goto done;
  cudaEventRecord(e1, nullptr);
  if (cudaDeviceSynchronize() != cudaSuccess) goto done;
  cudaEventElapsedTime(&ms, e0, e1);
  result[0] = result[1] = result[2] = 0.0;
  result[3] = ms;
  rc = 0;
done:
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (A) cudaFree(A);
  if (B) cudaFree(B);
  if (C) cudaFree(C);
  return rc;
}

// Grouped products against single products: nprob seeded operand pairs, each product computed
// alone and then all of them in one grouped launch, twice (each at the tile width that its number of
// tiles picks); result = [max |C_group - C_single| over the problems, error flag].
int selftest_gemm_group(int n, int prec, int mode, int nprob, double* result) {
  if (n % 128 || n <= 0 || nprob < 2 || nprob > kMaxGroup || !is_split_prec(prec)) return -1;
  const int esz = operand_bytes(prec);
  const bool single = mode >= 4;
  const int sym = single ? mode - 4 : mode;
  if (sym < 0 || sym > 2) return -1;
  EngineSplit eng(prec);
  const size_t cnt = (size_t)n * n;
  std::vector<SplitMat> A(nprob), B(nprob), C(nprob), R(nprob);
  double *tmp = nullptr, *out = nullptr;
  float* scal = nullptr;
  int rc = -2;
  std::vector<double> worst(1, 0.0);
  if (cudaMalloc((void**)&tmp, cnt * 8) || cudaMalloc((void**)&out, 8) || cudaMalloc((void**)&scal, sizeof(float)) ||
      cudaMemcpy(scal, &kUnitScale, sizeof(float), cudaMemcpyHostToDevice))
    goto done;
  for (int i = 0; i < nprob; ++i) {
    if (alloc_split(A[i], n, esz, scal, kF, nullptr) || alloc_split(B[i], n, esz, scal, kF, nullptr) ||
        alloc_split(C[i], n, esz, scal, kF, nullptr) || alloc_split(R[i], n, esz, scal, kF, nullptr))
      goto done;
    fill_random_kernel<<<nblk(cnt), 256>>>(cnt, n, 101 + 7 * i, 0, tmp);
    note_launch();
    to_f32_kernel<<<nblk(cnt), 256>>>(cnt, tmp, A[i].f);
    note_launch();
    fill_random_kernel<<<nblk(cnt), 256>>>(cnt, n, 203 + 11 * i, sym, tmp);
    note_launch();
    to_f32_kernel<<<nblk(cnt), 256>>>(cnt, tmp, B[i].f);
    note_launch();
    if (eng.operands(nullptr, A[i], n) || eng.operands(nullptr, B[i], n)) goto done;
  }
  {
    Epi ep;
    ep.pairs = (sym == 2) ? 2 : 1;
    ep.nseg = single ? 1 : 3;
    ep.alpha = 0.75f;
    for (int i = 0; i < nprob; ++i)
      if (eng.gemm(nullptr, n, {&A[i], &B[i], &R[i], ep, nullptr}, sym != 0)) goto done;
    std::vector<EngineSplit::GemmOp> ops;
    for (int i = 0; i < nprob; ++i) ops.push_back({&A[i], &B[i], &C[i], ep, nullptr});
    for (int rep = 0; rep < 2; ++rep) {   // the second launch reads the table that the first one built
      if (eng.gemm_group(nullptr, n, ops, sym != 0)) goto done;
      for (int i = 0; i < nprob; ++i) {
        if (cudaMemset(out, 0, 8)) goto done;
        diff_f32_kernel<<<304, 256>>>(cnt, C[i].f, R[i].f, out);
        note_launch();
        double h = 0.0;
        if (cudaMemcpy(&h, out, 8, cudaMemcpyDeviceToHost)) goto done;
        worst[0] = std::max(worst[0], h);
      }
    }
  }
  if (cudaDeviceSynchronize() != cudaSuccess) goto done;
  {
    int herr = 0;
    cudaMemcpy(&herr, eng.err_, sizeof(int), cudaMemcpyDeviceToHost);
    result[0] = worst[0];
    result[1] = herr;
    rc = 0;
  }
done:
  for (int i = 0; i < nprob; ++i) {
    free_split(A[i]);
    free_split(B[i]);
    free_split(C[i]);
    free_split(R[i]);
  }
  if (tmp) cudaFree(tmp);
  if (out) cudaFree(out);
  if (scal) cudaFree(scal);
  return rc;
}

// Returns 0 on success and writes [max |C_tc - C_ref|, max |C_ref|, error flag, ms per product].
int selftest_gemm(int n, int prec, int sym, double* result) {
  if (prec == 0 && n % 128 == 0 && n > 0 && sym >= 0 && sym <= 1) return selftest_gemm_f64(n, sym, result);
  if (n % 128 || n <= 0 || !is_split_prec(prec)) return -1;
  const int esz = operand_bytes(prec);
  const bool single = sym >= 4;   // one product of the hi operands only, as in the single-product chains
  if (single) sym -= 4;
  if (sym < 0 || sym > 2) return -1;
  EngineSplit eng(prec);
  const size_t cnt = (size_t)n * n;
  double *A = nullptr, *B = nullptr, *Cref = nullptr, *Cref2 = nullptr, *out = nullptr;
  const bool pair = (sym == 2);   // C = A B^T + B A^T
  float* scal = nullptr;
  SplitMat sa, sb, sc;
  cudaStream_t s = nullptr;
  int rc = -2;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  float ms = 0.f;
  if (cudaMalloc((void**)&A, cnt * 8) || cudaMalloc((void**)&B, cnt * 8) || cudaMalloc((void**)&Cref, cnt * 8) ||
      cudaMalloc((void**)&out, 8) || cudaMalloc((void**)&scal, sizeof(float)) ||
      (pair && cudaMalloc((void**)&Cref2, cnt * 8)))
    goto done;
  cudaMemcpy(scal, &kUnitScale, sizeof(float), cudaMemcpyHostToDevice);
  if (alloc_split(sa, n, esz, scal, kF, s) || alloc_split(sb, n, esz, scal, kF, s) ||
      alloc_split(sc, n, esz, scal, kF, s))
    goto done;
  fill_random_kernel<<<nblk(cnt), 256>>>(cnt, n, 11, 0, A);
  note_launch();
  fill_random_kernel<<<nblk(cnt), 256>>>(cnt, n, 23, sym, B);
  note_launch();
  to_f32_kernel<<<nblk(cnt), 256>>>(cnt, A, sa.f);
  note_launch();
  to_f32_kernel<<<nblk(cnt), 256>>>(cnt, B, sb.f);
  note_launch();
  if (eng.operands(s, sa, n) || eng.operands(s, sb, n)) goto done;
  {
    EpiF64 e;
    if (gemm_f64_nt(s, n, n, n, A, n, B, n, Cref, n, e, sym == 1)) goto done;
    if (pair) {   // Cref2 = B A^T + A B^T
      EpiF64 e2;
      e2.E = Cref;
      e2.lde = n;
      e2.beta = 1.0;
      if (gemm_f64_nt(s, n, n, n, B, n, A, n, Cref2, n, e2, false)) goto done;
    }
  }
  cudaEventCreate(&e0);
  cudaEventCreate(&e1);
  {
    Epi ep;
    ep.pairs = pair ? 2 : 1;
    ep.nseg = single ? 1 : 3;
    if (eng.gemm(s, n, {&sa, &sb, &sc, ep, nullptr}, sym != 0)) goto done;
    cudaEventRecord(e0, s);
    for (int r = 0; r < 5; ++r)
      if (eng.gemm(s, n, {&sa, &sb, &sc, ep, nullptr}, sym != 0)) goto done;
  }
  cudaEventRecord(e1, s);
  if (cudaDeviceSynchronize() != cudaSuccess) goto done;
  cudaEventElapsedTime(&ms, e0, e1);
  cudaMemset(out, 0, 8);
  max_abs_diff_kernel<<<304, 256>>>(cnt, sc.f, pair ? Cref2 : Cref, out);
  note_launch();
  if (cudaDeviceSynchronize() != cudaSuccess) goto done;
  {
    double h[1];
    int herr = 0;
    cudaMemcpy(h, out, 8, cudaMemcpyDeviceToHost);
    cudaMemcpy(&herr, eng.err_, sizeof(int), cudaMemcpyDeviceToHost);
    result[0] = h[0];
    result[1] = 0.0;
    result[2] = herr;
    result[3] = ms / 5.0;
    rc = 0;
  }
done:
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  free_split(sa);
  free_split(sb);
  free_split(sc);
  if (A) cudaFree(A);
  if (B) cudaFree(B);
  if (Cref) cudaFree(Cref);
  if (Cref2) cudaFree(Cref2);
  if (out) cudaFree(out);
  if (scal) cudaFree(scal);
  return rc;
}

}  // namespace xl
