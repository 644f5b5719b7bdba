// FP64 matrix products of the plain-FP64 path: C = epi(A * B^T).
//
// GB300 executes two FP64 multiply-adds per SM and clock (1.26 TFLOP/s over 152
// SMs), so a product is bound by how evenly its multiply-adds spread over the
// SMs, and operand traffic hardly matters: an 8 x 8 tile needs 16 doubles per K
// step, 4 bytes a clock.  Tiles are therefore as small as the matrix asks for:
//   8 x 8    one tile per CTA, its K range split over four warps
//   16 x 16  four warps, 8 x 8 each
//   32 x 32  four warps, 16 x 16 each
//   64 x 64  256 threads, 4 x 4 outputs each
// With 64 x 64 tiles alone a product of n = 128 ran on three or four SMs (135 us;
// now 8 x 8 tiles, symmetric 7.8 us, dense 9.8) and a symmetric one of n = 512 on 36
// (530 us; now 119; launch included).
#include "internal.h"

namespace xl {
namespace {

constexpr int KC = 16;   // K values staged at a time (M, N and K are multiples of 16)

// upper-triangular tile index t of nt x nt tiles -> (bi, bj), bj >= bi
__device__ __forceinline__ void sym_tile(int t, int nt, int& bi, int& bj) {
  // row r starts at r nt - r (r - 1) / 2
  int r = (int)((2.0f * nt + 1.0f - sqrtf((2.0f * nt + 1.0f) * (2.0f * nt + 1.0f) - 8.0f * t)) * 0.5f);
  r = min(max(r, 0), nt - 1);
  while (r > 0 && t < r * nt - r * (r - 1) / 2) --r;
  while (r + 1 < nt && t >= (r + 1) * nt - (r + 1) * r / 2) ++r;
  bi = r;
  bj = r + t - (r * nt - r * (r - 1) / 2);
}

template <bool SYM>
__device__ __forceinline__ void store_c(const EpiF64& e, double* C, int ldc, int row, int col, bool diag_tile,
                                        double acc) {
  if (SYM && diag_tile && row > col) return;
  double v = e.alpha * acc;
  if (e.E) v += e.beta * e.E[(size_t)row * e.lde + col];
  if (row == col) {
    v += e.diag;
    if (e.dvec && row < e.ndvec) v += e.dvec_scale * e.dvec[row];
  }
  C[(size_t)row * ldc + col] = v;
  if (SYM && row != col) C[(size_t)col * ldc + row] = v;
}

// One problem of a batch: blockIdx.z moves every matrix by its stride.
struct F64Batch {
  size_t a = 0, b = 0, c = 0, e = 0;
};

// 8 x 8 tiles: warp w takes the K chunks w, w + 4, ..; lane l holds (l / 4, l % 4) and (l / 4, l % 4 + 4).
template <bool SYM>
__global__ void __launch_bounds__(128) gemm_f64_t8_kernel(int M, int N, int K, const double* A, int lda,
                                                          const double* B, int ldb, double* C, int ldc,
                                                          EpiF64 e, F64Batch st) {
  grid_wait();
  __shared__ double sa[4][8][KC + 1], sb[4][8][KC + 1];
  __shared__ double red[3][64];
  A += st.a * blockIdx.z;
  B += st.b * blockIdx.z;
  C += st.c * blockIdx.z;
  if (e.E) e.E += st.e * blockIdx.z;
  int bi, bj;
  if (SYM) {
    sym_tile(blockIdx.x, N / 8, bi, bj);
  } else {
    bi = blockIdx.x / (N / 8);
    bj = blockIdx.x % (N / 8);
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, r = lane >> 2, c = lane & 3;
  // a lane loads two 16-byte pieces of each operand chunk: row lr (and lr + 4), K values lk, lk + 1
  const int lr = lane >> 3, lk = (lane & 7) * 2;
  const double* Ab = A + (size_t)(bi * 8 + lr) * lda + lk;
  const double* Bb = B + (size_t)(bj * 8 + lr) * ldb + lk;
  const int nc = K / KC;
  double acc0 = 0.0, acc1 = 0.0;
  double2 pa[2], pb[2];
  auto fetch = [&](int ch) {
    const size_t k = (size_t)ch * KC;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      pa[q] = *reinterpret_cast<const double2*>(Ab + (size_t)4 * q * lda + k);
      pb[q] = *reinterpret_cast<const double2*>(Bb + (size_t)4 * q * ldb + k);
    }
  };
  if (w < nc) fetch(w);
  for (int ch = w; ch < nc; ch += 4) {
    __syncwarp();
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      sa[w][lr + 4 * q][lk] = pa[q].x;
      sa[w][lr + 4 * q][lk + 1] = pa[q].y;
      sb[w][lr + 4 * q][lk] = pb[q].x;
      sb[w][lr + 4 * q][lk + 1] = pb[q].y;
    }
    __syncwarp();
    if (ch + 4 < nc) fetch(ch + 4);
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      const double a = sa[w][r][k];
      acc0 = fma(a, sb[w][c][k], acc0);
      acc1 = fma(a, sb[w][c + 4][k], acc1);
    }
  }
  if (w > 0) {
    red[w - 1][2 * lane] = acc0;
    red[w - 1][2 * lane + 1] = acc1;
  }
  __syncthreads();
  if (w > 0) return;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    acc0 += red[q][2 * lane];
    acc1 += red[q][2 * lane + 1];
  }
  const int row = bi * 8 + r, col = bj * 8 + c;
  store_c<SYM>(e, C, ldc, row, col, bi == bj, acc0);
  store_c<SYM>(e, C, ldc, row, col + 4, bi == bj, acc1);
}

// T x T tiles (16 or 32), four warps in 2 x 2, each (T / 2)^2 outputs as 8 x 8 blocks of two per lane.
template <int T, bool SYM>
__global__ void __launch_bounds__(128) gemm_f64_t_kernel(int M, int N, int K, const double* A, int lda,
                                                         const double* B, int ldb, double* C, int ldc,
                                                         EpiF64 e, F64Batch st) {
  grid_wait();
  constexpr int NB = T / 16;              // 8 x 8 blocks per warp and dimension
  constexpr int PER = T * KC / 2 / 128;   // 16-byte pieces per thread, operand and chunk
  __shared__ double sa[2][T][KC + 1], sb[2][T][KC + 1];
  A += st.a * blockIdx.z;
  B += st.b * blockIdx.z;
  C += st.c * blockIdx.z;
  if (e.E) e.E += st.e * blockIdx.z;
  int bi, bj;
  const int nt = (N + T - 1) / T;   // rows past M and N are loaded and not stored
  if (SYM) {
    sym_tile(blockIdx.x, nt, bi, bj);
  } else {
    bi = blockIdx.x / nt;
    bj = blockIdx.x % nt;
  }
  const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
  const int r = (w >> 1) * (T / 2) + (lane >> 2), c = (w & 1) * (T / 2) + (lane & 3);
  const int nc = K / KC;
  double2 pa[PER], pb[PER];
  auto fetch = [&](int ch) {
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int el = tid + 128 * q, row = el >> 3, k = (el & 7) * 2;
      pa[q] = *reinterpret_cast<const double2*>(A + (size_t)(bi * T + row) * lda + ch * KC + k);
      pb[q] = *reinterpret_cast<const double2*>(B + (size_t)(bj * T + row) * ldb + ch * KC + k);
    }
  };
  double acc[NB][NB][2];
#pragma unroll
  for (int i = 0; i < NB; ++i)
#pragma unroll
    for (int j = 0; j < NB; ++j) acc[i][j][0] = acc[i][j][1] = 0.0;
  fetch(0);
  for (int ch = 0; ch < nc; ++ch) {
    const int b = ch & 1;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int el = tid + 128 * q, row = el >> 3, k = (el & 7) * 2;
      sa[b][row][k] = pa[q].x;
      sa[b][row][k + 1] = pa[q].y;
      sb[b][row][k] = pb[q].x;
      sb[b][row][k + 1] = pb[q].y;
    }
    __syncthreads();   // buffer b is written; the other one was read before the last barrier
    if (ch + 1 < nc) fetch(ch + 1);
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      double a[NB], x[NB][2];
#pragma unroll
      for (int i = 0; i < NB; ++i) a[i] = sa[b][r + 8 * i][k];
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        x[j][0] = sb[b][c + 8 * j][k];
        x[j][1] = sb[b][c + 8 * j + 4][k];
      }
#pragma unroll
      for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int j = 0; j < NB; ++j) {
          acc[i][j][0] = fma(a[i], x[j][0], acc[i][j][0]);
          acc[i][j][1] = fma(a[i], x[j][1], acc[i][j][1]);
        }
    }
  }
#pragma unroll
  for (int i = 0; i < NB; ++i)
#pragma unroll
    for (int j = 0; j < NB; ++j) {
      const int row = bi * T + r + 8 * i, col = bj * T + c + 8 * j;
      if (row >= M || col >= N) continue;   // a multiple of 8 each: col + 4 is inside with col
      store_c<SYM>(e, C, ldc, row, col, bi == bj, acc[i][j][0]);
      store_c<SYM>(e, C, ldc, row, col + 4, bi == bj, acc[i][j][1]);
    }
}

template <bool SYM>
__global__ void __launch_bounds__(256) gemm_f64_kernel(int M, int N, int K, const double* A,
                                                       int lda, const double* B, int ldb,
                                                       double* C, int ldc, EpiF64 e, F64Batch st) {
  grid_wait();
  constexpr int BM = 64, BN = 64, BK = KC;
  A += st.a * blockIdx.z;
  B += st.b * blockIdx.z;
  C += st.c * blockIdx.z;
  if (e.E) e.E += st.e * blockIdx.z;
  int bi, bj;
  const int nt = (N + BN - 1) / BN;
  if (SYM) {
    sym_tile(blockIdx.x, nt, bi, bj);
  } else {
    bi = blockIdx.x / nt;
    bj = blockIdx.x % nt;
  }
  __shared__ double As[BK][BM + 1];
  __shared__ double Bs[BK][BN + 1];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  double acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0;
  const double* Ab = A + (size_t)bi * BM * lda;
  const double* Bb = B + (size_t)bj * BN * ldb;
  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int el = tid + 256 * r, row = el >> 4, col = el & 15;
      As[col][row] = Ab[(size_t)row * lda + k0 + col];
      Bs[col][row] = Bb[(size_t)row * ldb + k0 + col];
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      double a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (bi * BM + 16 * i < M && bj * BN + 16 * j < N)
        store_c<SYM>(e, C, ldc, bi * BM + ty + 16 * i, bj * BN + tx + 16 * j, bi == bj, acc[i][j]);
}

// Tile edge of a product: the one with the least waves over the SMs times the tile's multiply-adds, with
// a few per cent for the staging of small tiles (they win where they fill the SMs: n = 128 to 640; from
// about n = 1500 on the waves even out and 64 x 64 runs at 99.6 % of the FP64 rate).
int pick_tile(int M, int N, bool sym, int batch) {
  const int edge[4] = {8, 16, 32, 64};
  const double over[4] = {1.06, 1.03, 1.01, 1.0};
  int best = 64;
  double least = 0.0;
  for (int i = 0; i < 4; ++i) {
    const long long nt = (N + edge[i] - 1) / edge[i];
    const long long tiles = batch * (sym ? nt * (nt + 1) / 2 : nt * ((M + edge[i] - 1) / edge[i]));
    const double c = (double)((tiles + 151) / 152) * edge[i] * edge[i] * over[i];
    if (least == 0.0 || c < least) {
      least = c;
      best = edge[i];
    }
  }
  return best;
}

template <bool SYM>
cudaError_t launch(cudaStream_t s, int tile, dim3 grid, int M, int N, int K, const double* A, int lda, const double* B, int ldb,
            double* C, int ldc, const EpiF64& e, const F64Batch& st) {
  switch (tile) {
    case 8:
      return launch_chained(s, grid, 128, 0, gemm_f64_t8_kernel<SYM>, M, N, K, A, lda, B, ldb, C, ldc, e, st);
    case 16:
      return launch_chained(s, grid, 128, 0, gemm_f64_t_kernel<16, SYM>, M, N, K, A, lda, B, ldb, C, ldc, e, st);
    case 32:
      return launch_chained(s, grid, 128, 0, gemm_f64_t_kernel<32, SYM>, M, N, K, A, lda, B, ldb, C, ldc, e, st);
    default:
      return launch_chained(s, grid, 256, 0, gemm_f64_kernel<SYM>, M, N, K, A, lda, B, ldb, C, ldc, e, st);
  }
}

}  // namespace

cudaError_t gemm_f64_nt(cudaStream_t s, int M, int N, int K, const double* A, int lda, const double* B,
                        int ldb, double* C, int ldc, const EpiF64& e, bool sym, int batch, size_t stA, size_t stB,
                        size_t stC, size_t stE) {
  if (M % 16 || N % 16 || K % KC || M <= 0 || N <= 0 || K <= 0 || batch < 1) return cudaErrorInvalidValue;
  if (sym && M != N) return cudaErrorInvalidValue;
  const int t = pick_tile(M, N, sym, batch);
  const long long nt = (N + t - 1) / t;
  const dim3 grid((unsigned)(sym ? nt * (nt + 1) / 2 : nt * ((M + t - 1) / t)), 1, (unsigned)batch);
  const F64Batch st{stA, stB, stC, stE};
  return sym ? launch<true>(s, t, grid, M, N, K, A, lda, B, ldb, C, ldc, e, st)
             : launch<false>(s, t, grid, M, N, K, A, lda, B, ldb, C, ldc, e, st);
}

}  // namespace xl
