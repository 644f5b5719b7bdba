// Tensor-core split-precision product (gemm_tc.cu) interface.
#pragma once
#include <cstdint>
#include <vector>

#include <cuda.h>
#include <cuda_runtime.h>

namespace xl {

// Where a product's result goes; what is null is not written.  f: FP32 value, d: double-float value,
// hi (and lo): tensor-core operands of the value times *scale.
struct TcOut {
  float* f = nullptr;
  float2* d = nullptr;
  void* hi = nullptr;
  void* lo = nullptr;
  const float* scale = nullptr;
};

struct TcArgs {
  int K = 0;                      // inner dimension (set by gemm_tc)
  int n = 0;                      // matrix size (set by gemm_tc)
  int split_acc = 0;              // one-CTA-per-tile kernel: 1 = the hi*hi K blocks split over both
                                  // accumulators (below)
  int chunk_kb = 0;               // split products: the hi*hi sum is accumulated in chunks of this many
                                  // K blocks, added up in FP32 (0: one chunk)
  int nseg = 3;                   // 1: hi only; 3: hi*hi + hi*lo + lo*hi
  int pairs = 1;                  // 2: C = A B^T + B A^T (the swapped pair as a second K range)
  int sym = 0;                    // symmetric output (upper tiles, mirrored)
  int fmt = 0;                    // operand type: 0 FP16, 1 BF16 (kind::f16), 2 TF32 (kind::tf32,
                                  // FP32 words; persistent kernel only)
  int tiles_n = 0;                // set by gemm_tc
  const int* tile_list = nullptr; // set by gemm_tc
  float alpha = 1.0f;             // v = alpha acc / (sa sb) + beta E + beta2 E2 + diag I
  const float* E = nullptr;       //     + dvec_scale diag(dvec)
  float beta = 0.0f;
  const float* E2 = nullptr;
  float beta2 = 0.0f;
  const float2* E64 = nullptr;    // out.d: v + beta64 E64 as a double-float (beta64 a power of two,
  float beta64 = 0.0f;            // so that beta64 E64 is exact)
  float diag = 0.0f;
  const double* dvec = nullptr;
  int ndvec = 0;
  float dvec_scale = 1.0f;
  TcOut out;
  TcOut out2;                     // a second result va v + vb E (f, hi, lo; E symmetric)
  float va = 0.0f, vb = 0.0f;
  int ldc = 0;
  const float* sa = nullptr;      // operand scales (device scalars)
  const float* sb = nullptr;
  int* err = nullptr;             // set non-zero when a bounded wait gives up
};

// One problem of a grouped product launch, in device memory: its tensor maps (A hi, A lo, B hi,
// B lo, and the second pair's A2 hi, A2 lo, B2 hi, B2 lo) and its epilogue arguments.  The
// problems of a group share n, the segment and pair counts, the symmetric mode and the operand
// type; they differ in their matrices and scalars.
struct TcEntry {   // CUtensorMap's own alignment (64 bytes) aligns every entry
  CUtensorMap map[8];
  TcArgs args;
};

// One problem of a grouped product: operands and its epilogue arguments (n, K, nseg, pairs,
// sym, fmt, chunk_kb and err come from the launch's shared arguments).
struct TcProblem {
  const void *Ahi = nullptr, *Alo = nullptr, *Bhi = nullptr, *Blo = nullptr;   // operand arrays (n x n, row-major)
  // the second pair of pairs = 2: C = A B^T + A2 B2^T.  Null: B and A.  The scales of A2 and B2 multiply to
  // those of A and B.
  const void *A2hi = nullptr, *A2lo = nullptr, *B2hi = nullptr, *B2lo = nullptr;
  TcArgs epi;
};

// Device tile lists of the symmetric-output products of one size n (pairs of ints (tm, tn)):
// 128 x w tiles for the widths w = 32, 64, 128 and 256 (the last where n is a multiple of 256), and
// 256 x 256 tiles of the two-SM products (n a multiple of 256; null: not used for this size).
constexpr int kTcWidths = 4;
constexpr int tc_width(int i) { return 32 << i; }
struct TcTiles {
  const int* sym[kTcWidths] = {nullptr, nullptr, nullptr, nullptr};
  int nsym[kTcWidths] = {0, 0, 0, 0};
  const int* pair = nullptr;
  int npair = 0;
};

// n x n product (n a multiple of 128); the symmetric tile lists come from tc_sym_tiles and
// tc_sym_tiles_pair.
cudaError_t gemm_tc(cudaStream_t s, int n, const TcProblem& prob, const TcTiles& tiles);
// Grouped product: the problems' tiles in one persistent launch (one-SM kernel).  The device
// table of each distinct problem list is built once and kept in `cache` (key: the table's
// bytes), so repeated groups upload nothing.
struct TcGroupCache;
TcGroupCache* tc_group_cache_new();
void tc_group_cache_free(TcGroupCache* c);
cudaError_t gemm_tc_group(cudaStream_t s, int n, const TcProblem* probs, int nprob, TcArgs shared,
                          const TcTiles& tiles, TcGroupCache* cache);
std::vector<int> tc_sym_tiles(int n, int bn);
std::vector<int> tc_sym_tiles_pair(int n);
void tc_forget_maps(const void* base);

}  // namespace xl
