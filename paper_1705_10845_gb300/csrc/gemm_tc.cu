// Split-precision tensor-core products for sm_103a (tcgen05 + TMEM + TMA).
//
// C = epi( sum_seg A_seg B_seg^T ) with 16-bit operands (FP16 or BF16) and an
// FP32 accumulation in tensor memory.  A split product uses three K segments,
// A_hi B_hi + A_hi B_lo + A_lo B_hi (one, A_hi B_hi, for single-product
// chains); the operands carry power-of-two scales that the epilogue removes.
//
// The default kernel is persistent: one CTA per SM walks the 128 x BN output
// tiles, BN = 32 to 256 by size (pick_width).  Warp 0 issues TMA loads
// (128-byte swizzle, K-major) into a ring guarded by mbarriers; one thread of
// warp 1 issues tcgen05.mma (M = 128, N = BN, K = 16) per 32-byte K step; the
// epilogue warps read finished chunks of the sum with tcgen05.ld, add them up in
// registers, and write the value and the operands (hi, lo) that the next
// products read.  Two others are kept beside it: one tile per CTA
// (XLBOMD_GEMM=classic) and a two-SM form (XLBOMD_GEMM=pair).
//
// Against the version that wrote FP32 values, raised each matrix's maximum
// and left the operands to a conversion pass (memset, product, conversion; 128- or
// 256-wide tiles), per product: n = 128 27 -> 8.5 us, 256 44 -> 10.6, 640 37 -> 16, 1024
// 60 -> 22, 2048 82 -> 60 (symmetric 83 -> 48), 8192 2.31 -> 2.30 ms with sums half as long.
//
// The tensor core adds each K = 16 step into its FP32 accumulator with
// truncation, so a small term added to a large accumulator loses bits.  The
// hi*hi segment and the two correction segments (hi*lo, lo*hi, about 2^-11
// smaller) therefore never share an accumulator.  A pair product (pairs = 2) adds
// the swapped operands as a second K range, C = A B^T + B A^T.  Every mbarrier
// wait is bounded: on timeout the kernel records an error code and leaves its
// loops, waits (again bounded) for the copies and MMAs it has in flight, so that
// none of them lands in the shared memory or TMEM of the CTA that comes next, and
// releases TMEM.
//
// TF32 operands (fmt = 2, persistent kernel only) are FP32 words whose low 13
// mantissa bits are zero.  A 128-byte swizzle row then holds 32 elements, and
// each tcgen05.mma of kind::tf32 (K = 8) takes the same 32-byte step.  So the
// ring's stage bytes, the shared-memory descriptors and the per-stage MMA
// count stay as they are.  Only the K-block width (32 elements), the tensor
// map's element type and the instruction kind change.
#include <cuda.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <cstdlib>
#include <mutex>
#include <string>
#include <unordered_map>

#include "operand.cuh"
#include "precision.h"
#include "ring.h"
#include "tc.h"

namespace xl {
namespace {

constexpr int BM = 128;
constexpr int BK = 64;           // 64 x 16-bit = 128 bytes: one swizzle row
constexpr int STAGES = 4;        // one-CTA-per-tile kernel
constexpr int A_BYTES = BM * BK * 2;
constexpr int kOnceMaxN = 3072;  // largest size (multiple of 256) of the narrow tiles
constexpr int kWaitLimit = 1 << 24;
constexpr int kGroupM = 16;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

// Bounded wait for the completion of the phase with the given parity (the epilogue warps'
// waits: each try may suspend the thread for a hardware-chosen time).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  for (int it = 0; it < kWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// The same without suspending (mbarrier.test_wait in a bounded spin): the waits of the producer
// and MMA threads, which hand the operand ring's stages to each other (MMA completion -> empty
// -> producer -> full -> MMA thread).  With the default suspension those hand-offs cost about
// 20 % of a product (n = 8192 split product: 2.46 ms with the hand-off and no operand loads at
// all, 2.01 ms with neither), and the spin closes that gap (no loads: 1.92 ms; with loads 2.21
// against 2.26 ms with a 20 ns suspend hint).  The epilogue warps keep the suspending wait:
// polling from them would take issue slots from the two single-thread loops on the
// sub-partitions they share.
__device__ __forceinline__ bool mbar_wait_fast(uint64_t* bar, uint32_t parity) {
  const uint32_t a = smem_u32(bar);
  for (int it = 0; it < (kWaitLimit << 4); ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// After a wait that gave up: the copies that the ring's producer has in flight (each wait bounded; the first
// that gives up ends it).
__device__ __forceinline__ void drain_ring(uint64_t* full, int stages, uint32_t slot, uint32_t ph, bool first) {
  for (int s = 0; s < stages; ++s) {
    const int u = ring_last_use(slot, ph, first, s);
    if (u >= 0 && !mbar_wait(&full[s], (uint32_t)u)) return;
  }
}

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<uint64_t>(p)));
}

// A tensor map written to global memory by the host (grouped launches) reaches the TMA unit
// through the tensormap proxy: acquire it before its first use in the kernel.
__device__ __forceinline__ void tensormap_acquire(const CUtensorMap* map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.sys [%0], 128;" ::"l"(reinterpret_cast<uint64_t>(map))
               : "memory");
}

__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (SBO), descriptor version 1.
__device__ __forceinline__ uint64_t smem_desc(const void* p) {
  const uint32_t a = smem_u32(p);
  uint64_t d = 0;
  d |= (uint64_t)((a >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;              // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;    // stride byte offset
  d |= (uint64_t)1 << 46;              // version
  d |= (uint64_t)2 << 61;              // 128-byte swizzle
  return d;
}

// Instruction descriptor of kind::f16 / kind::tf32: D = F32, A/B = F16 (0) or BF16 (1) under
// kind::f16, TF32 (2) under kind::tf32, both K-major, M x N.
__host__ __device__ constexpr uint32_t instr_desc_m(int m, int bn, int ab_fmt) {
  return (1u << 4) | ((uint32_t)ab_fmt << 7) | ((uint32_t)ab_fmt << 10) | ((uint32_t)(bn >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}
__host__ __device__ constexpr uint32_t instr_desc(int bn, int ab_fmt) { return instr_desc_m(BM, bn, ab_fmt); }

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  // r tied to the wait: no use of the loaded registers is scheduled before it
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31])::"memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 64 columns of this warp's 32 lanes, without waiting (tcgen05.wait::ld before use)
__device__ __forceinline__ void tmem_ld64_nowait(uint32_t taddr, uint32_t (&r)[64]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63}, [%64];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]), "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]), "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]), "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]), "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr));
}

// Wait for this thread's tcgen05.ld results; r is tied to the wait so that no use of the loaded
// registers is scheduled before it.
__device__ __forceinline__ void tmem_wait_ld64(uint32_t (&r)[64]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]), "+r"(r[32]), "+r"(r[33]), "+r"(r[34]), "+r"(r[35]), "+r"(r[36]), "+r"(r[37]), "+r"(r[38]), "+r"(r[39]), "+r"(r[40]), "+r"(r[41]), "+r"(r[42]), "+r"(r[43]), "+r"(r[44]), "+r"(r[45]), "+r"(r[46]), "+r"(r[47]), "+r"(r[48]), "+r"(r[49]), "+r"(r[50]), "+r"(r[51]), "+r"(r[52]), "+r"(r[53]), "+r"(r[54]), "+r"(r[55]), "+r"(r[56]), "+r"(r[57]), "+r"(r[58]), "+r"(r[59]), "+r"(r[60]), "+r"(r[61]), "+r"(r[62]), "+r"(r[63])::"memory");
}

// Orders the uses of r after the preceding tcgen05.wait::ld (volatile asm statements keep their order).
__device__ __forceinline__ void tmem_after_wait64(uint32_t (&r)[64]) { asm volatile("" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15]), "+r"(r[16]), "+r"(r[17]), "+r"(r[18]), "+r"(r[19]), "+r"(r[20]), "+r"(r[21]), "+r"(r[22]), "+r"(r[23]), "+r"(r[24]), "+r"(r[25]), "+r"(r[26]), "+r"(r[27]), "+r"(r[28]), "+r"(r[29]), "+r"(r[30]), "+r"(r[31]), "+r"(r[32]), "+r"(r[33]), "+r"(r[34]), "+r"(r[35]), "+r"(r[36]), "+r"(r[37]), "+r"(r[38]), "+r"(r[39]), "+r"(r[40]), "+r"(r[41]), "+r"(r[42]), "+r"(r[43]), "+r"(r[44]), "+r"(r[45]), "+r"(r[46]), "+r"(r[47]), "+r"(r[48]), "+r"(r[49]), "+r"(r[50]), "+r"(r[51]), "+r"(r[52]), "+r"(r[53]), "+r"(r[54]), "+r"(r[55]), "+r"(r[56]), "+r"(r[57]), "+r"(r[58]), "+r"(r[59]), "+r"(r[60]), "+r"(r[61]), "+r"(r[62]), "+r"(r[63])); }

__device__ __forceinline__ void tmem_st64(uint32_t taddr, const uint32_t (&v)[64]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x64.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32, %33, %34, %35, %36, %37, %38, %39, %40, %41, %42, %43, %44, %45, %46, %47, %48, %49, %50, %51, %52, %53, %54, %55, %56, %57, %58, %59, %60, %61, %62, %63, %64};" ::"r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]), "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15]), "r"(v[16]), "r"(v[17]), "r"(v[18]), "r"(v[19]), "r"(v[20]), "r"(v[21]), "r"(v[22]), "r"(v[23]), "r"(v[24]), "r"(v[25]), "r"(v[26]), "r"(v[27]), "r"(v[28]), "r"(v[29]), "r"(v[30]), "r"(v[31]), "r"(v[32]), "r"(v[33]), "r"(v[34]), "r"(v[35]), "r"(v[36]), "r"(v[37]), "r"(v[38]), "r"(v[39]), "r"(v[40]), "r"(v[41]), "r"(v[42]), "r"(v[43]), "r"(v[44]), "r"(v[45]), "r"(v[46]), "r"(v[47]), "r"(v[48]), "r"(v[49]), "r"(v[50]), "r"(v[51]), "r"(v[52]), "r"(v[53]), "r"(v[54]), "r"(v[55]), "r"(v[56]), "r"(v[57]), "r"(v[58]), "r"(v[59]), "r"(v[60]), "r"(v[61]), "r"(v[62]), "r"(v[63]) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Output tile of tile id: from the symmetric tile list, or the grouped raster (GROUP_M row
// panels at a time, so that the CTAs in flight share their A and B panels in L2).  False for
// a tile outside the matrix (a bad tile list), which is reported and never stored.
__device__ __forceinline__ bool tile_coords(const TcArgs& a, int id, int& tm, int& tn) {
  if (a.tile_list) {
    tm = a.tile_list[2 * id];
    tn = a.tile_list[2 * id + 1];
  } else {
    const int tiles_m = a.n / BM;
    const int per_group = kGroupM * a.tiles_n;
    const int g = id / per_group, r = id % per_group;
    const int first = g * kGroupM;
    const int gm = min(tiles_m - first, kGroupM);
    tm = first + r % gm;
    tn = r / gm;
  }
  return tm >= 0 && tm < a.n / BM && tn >= 0 && tn < a.tiles_n;
}

// The K blocks of a tile run as a few segments, each one operand pair pr (0: A B^T, 1: the
// swapped pair B A^T) and split part kind (0 = hi*hi, 1 = hi*lo, 2 = lo*hi) over K blocks
// [k0, k1).  Default order: the hi*hi segments of every pair (accumulator 0), then the
// corrections (accumulator 1).  split_acc (large n): the first half of the hi*hi K blocks
// (accumulator 0), the corrections into accumulator 1 while it is still small, then the second
// half of the hi*hi K blocks on top of accumulator 1 -- the tensor core truncates as it
// accumulates, so each large sum is half as long.  Accumulator 1 starts at K block acc1_start.
struct KSeg {
  int seg, kidx, k1, pr, kind;
};

__device__ __forceinline__ void kseg_decode(const TcArgs& a, int nk, KSeg& q) {
  const int P = a.pairs, NC = (a.nseg - 1) * a.pairs;   // hi*hi pairs, correction segments
  int k0 = 0;
  q.k1 = nk;
  if (!a.split_acc) {
    if (q.seg < P) {
      q.pr = q.seg;
      q.kind = 0;
    } else {
      const int r = q.seg - P;
      q.pr = r >> 1;
      q.kind = 1 + (r & 1);
    }
  } else if (q.seg == 0 || q.seg > NC) {
    const bool second = q.seg > NC;
    q.kind = 0;
    if (P == 2) {
      q.pr = second ? 1 : 0;
    } else {
      q.pr = 0;
      k0 = second ? nk / 2 : 0;
      q.k1 = second ? nk : nk / 2;
    }
  } else {
    const int r = q.seg - 1;
    q.pr = r >> 1;
    q.kind = 1 + (r & 1);
  }
  q.kidx = k0;
}

__device__ __forceinline__ void kseg_begin(const TcArgs& a, int nk, KSeg& q) {
  q.seg = 0;
  kseg_decode(a, nk, q);
}

__device__ __forceinline__ void kseg_next(const TcArgs& a, int nk, KSeg& q) {
  if (++q.kidx == q.k1) {
    ++q.seg;
    kseg_decode(a, nk, q);
  }
}

__device__ __forceinline__ int acc1_start(const TcArgs& a, int nk) {
  return a.split_acc ? a.pairs * nk / 2 : a.pairs * nk;
}

// L2 prefetch of the side inputs of the 128 x BN tile (tm, tn) by nt epilogue threads
template <int BN, typename Args>
__device__ __forceinline__ void prefetch_sides(const Args& a, int tm, int tn, int t, int nt) {
  const float* fsides[2] = {a.E, a.E2};
  for (int k = 0; k < 2; ++k)
    if (fsides[k])
      for (int i = t; i < BM * (BN / 32); i += nt)
        prefetch_l2(fsides[k] + (size_t)(tm * BM + i / (BN / 32)) * a.ldc + tn * BN + (i % (BN / 32)) * 32);
  if (a.E64)
    for (int i = t; i < BM * (BN / 16); i += nt)
      prefetch_l2(a.E64 + (size_t)(tm * BM + i / (BN / 16)) * a.ldc + tn * BN + (i % (BN / 16)) * 16);
}

// a + b for a double-float a and a float b (Knuth two-sum, then renormalise)
__device__ __forceinline__ float2 df_add(float2 a, float b) {
  const float s = a.x + b;
  const float bb = s - a.x;
  const float err = (a.x - (s - bb)) + (b - bb) + a.y;
  const float hi = s + err;
  return make_float2(hi, err - (hi - s));
}

// The epilogue's arguments in registers.  (Read through a reference to the kernel parameter or to a
// grouped launch's table they are loaded again after every store: 4 us per 32 x 32 chunk.)
struct EpiRegs {
  const float *E, *E2;
  const float2* E64;
  const double* dvec;
  float beta, beta2, beta64, diag, dvec_scale, va, vb, inv, so, so2;
  float *f, *f2;
  float2* d;
  void *hi, *lo, *hi2, *lo2;
  int ldc, ndvec, fmt;
  bool sym;
};

__device__ __forceinline__ EpiRegs load_epi(const TcArgs& a) {
  EpiRegs e;
  e.E = a.E;
  e.E2 = a.E2;
  e.E64 = a.E64;
  e.dvec = a.dvec;
  e.beta = a.beta;
  e.beta2 = a.beta2;
  e.beta64 = a.beta64;
  e.diag = a.diag;
  e.dvec_scale = a.dvec_scale;
  e.va = a.va;
  e.vb = a.vb;
  e.inv = a.alpha / (*a.sa * *a.sb);
  e.f = a.out.f;
  e.d = a.out.d;
  e.hi = a.out.hi;
  e.lo = a.out.lo;
  e.so = a.out.hi ? *a.out.scale : 0.0f;
  e.f2 = a.out2.f;
  e.hi2 = a.out2.hi;
  e.lo2 = a.out2.lo;
  e.so2 = a.out2.hi ? *a.out2.scale : 0.0f;
  e.ldc = a.ldc;
  e.ndvec = a.ndvec;
  e.fmt = a.fmt;
  e.sym = a.sym != 0;
  return e;
}

// 4 x 4 values x + xl: four neighbouring columns at element i and every st-th one after it.
template <int FMT>
__device__ __forceinline__ void store_operands(void* hi, void* lo, float s, size_t i, size_t st, const float (&x)[4][4],
                                               const float (&xl)[4][4]) {
  if (lo) {
#pragma unroll
    for (int q = 0; q < 4; ++q) store_operand4<FMT>(hi, lo, i + q * st, s, x[q], xl[q]);
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q) store_operand4<FMT>(hi, nullptr, i + q * st, s, x[q], xl[q]);
  }
}

template <bool TF32>
__device__ __forceinline__ void store_out(float* f, float2* d, void* hi, void* lo, int fmt, float s, size_t i, size_t st,
                                          const float (&x)[4][4], const float (&xl)[4][4]) {
  if (f) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<float4*>(f + i + q * st) = make_float4(x[q][0], x[q][1], x[q][2], x[q][3]);
  }
  if (d) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      float4* p = reinterpret_cast<float4*>(d + i + q * st);
      p[0] = make_float4(x[q][0], xl[q][0], x[q][1], xl[q][1]);
      p[1] = make_float4(x[q][2], xl[q][2], x[q][3], xl[q][3]);
    }
  }
  if (hi) {
    if constexpr (TF32)
      store_operands<2>(hi, lo, s, i, st, x, xl);
    else if (fmt)
      store_operands<1>(hi, lo, s, i, st, x, xl);
    else
      store_operands<0>(hi, lo, s, i, st, x, xl);
  }
}

// 4 x 4 values of a side input; on a diagonal chunk from its upper triangle.
__device__ __forceinline__ void load_side(float (&e)[4][4], const float* E, size_t i, size_t st, bool dg,
                                          int row, int col, int ldc) {
  if (!dg) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 w = *reinterpret_cast<const float4*>(E + i + q * st);
      e[q][0] = w.x;
      e[q][1] = w.y;
      e[q][2] = w.z;
      e[q][3] = w.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int r = row + 4 * q, c = col + k;
        e[q][k] = E[(size_t)min(r, c) * ldc + max(r, c)];
      }
  }
}

__device__ __forceinline__ void axpy44(float (&x)[4][4], float b, const float (&e)[4][4]) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k) x[q][k] += b * e[q][k];
}

// Epilogue of one 32 x 32 chunk at (row0, col0), whose scaled sums are in the warp's staging tile t.  A
// lane takes columns 4 (l % 8) .. + 3 of rows l / 8, + 4, + 8, + 12 (and the same of the lower 16 rows), so
// that every side input is read and every result written in 16-byte pieces of whole rows (8 bytes of
// 16-bit operands), and each option is decided once per 16 values: with a branch per value group the
// chunk took 5 to 10 us of a small product's 20.  A symmetric product skips chunks below the
// diagonal and writes the others a second time, transposed: FP32 results through the staging tile,
// double-float results (two words, for which the tile has no room) read back from where this warp
// has just stored them.  Diagonal chunks take their upper triangle for both halves.
template <bool TF32>
__device__ __forceinline__ void epilogue_chunk(const EpiRegs& a, int row0, int col0, int lane, float (*t)[33]) {
  const bool dg = a.sym && col0 == row0;
  const int lr = lane >> 3, lc = (lane & 7) * 4;
  const size_t st = 4 * (size_t)a.ldc;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int r0 = 16 * h + lr, row = row0 + r0, col = col0 + lc;
    const size_t i = (size_t)row * a.ldc + col;
    float x[4][4], xl[4][4], e[4][4], e2[4][4];
    if (a.E) load_side(e, a.E, i, st, dg, row, col, a.ldc);
    if (a.E2) load_side(e2, a.E2, i, st, dg, row, col, a.ldc);
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < 4; ++k) xl[q][k] = 0.0f;
    if (!dg) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) x[q][k] = t[r0 + 4 * q][lc + k];
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int r = r0 + 4 * q, c = lc + k;
          x[q][k] = t[min(r, c)][max(r, c)];
        }
    }
    if (a.E && a.beta != 0.0f) axpy44(x, a.beta, e);
    if (a.E2) axpy44(x, a.beta2, e2);
    if (row0 == col0 && (a.diag != 0.0f || a.dvec)) {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = row + 4 * q, dc = r - col;
        if (dc >= 0 && dc < 4) {
          float dd = a.diag;
          if (a.dvec && r < a.ndvec) dd += a.dvec_scale * (float)a.dvec[r];
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k == dc) x[q][k] += dd;
        }
      }
    }
    if (a.hi2) {
      float y[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) y[q][k] = a.va * x[q][k];
      axpy44(y, a.vb, e);
      store_out<TF32>(a.f2, nullptr, a.hi2, a.lo2, a.fmt, a.so2, i, st, y, xl);
    }
    if (a.E64) {
      if (!dg) {
        float4 w[4][2];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4* p = reinterpret_cast<const float4*>(a.E64 + i + q * st);
          w[q][0] = p[0];
          w[q][1] = p[1];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float eh[4] = {w[q][0].x, w[q][0].z, w[q][1].x, w[q][1].z};
          const float el[4] = {w[q][0].y, w[q][0].w, w[q][1].y, w[q][1].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float2 z = df_add(make_float2(a.beta64 * eh[k], a.beta64 * el[k]), x[q][k]);
            x[q][k] = z.x;
            xl[q][k] = z.y;
          }
        }
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const int r = row + 4 * q, c = col + k;
            const float2 e = a.E64[(size_t)min(r, c) * a.ldc + max(r, c)];
            const float2 z = df_add(make_float2(a.beta64 * e.x, a.beta64 * e.y), x[q][k]);
            x[q][k] = z.x;
            xl[q][k] = z.y;
          }
      }
    }
    if (a.sym && !dg && !a.d) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) t[r0 + 4 * q][lc + k] = x[q][k];
    }
    store_out<TF32>(a.f, a.d, a.hi, a.lo, a.fmt, a.so, i, st, x, xl);
  }
  __syncwarp();
  if (!a.sym || dg) return;
#pragma unroll 1
  for (int h = 0; h < 2; ++h) {
    const int c0 = 16 * h + lr;   // output rows col0 + c0, + 4, ..; columns row0 + lc ..
    const size_t i = (size_t)(col0 + c0) * a.ldc + row0 + lc;
    float x[4][4], xl[4][4];
    if (a.d) {
      float2 z[4][4];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) z[q][k] = a.d[(size_t)(row0 + lc + k) * a.ldc + col0 + c0 + 4 * q];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          x[q][k] = z[q][k].x;
          xl[q][k] = z[q][k].y;
        }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          x[q][k] = t[lc + k][c0 + 4 * q];
          xl[q][k] = 0.0f;
        }
    }
    if (a.hi2) {
      float y[4][4], e[4][4];
      load_side(e, a.E, i, st, false, 0, 0, a.ldc);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int k = 0; k < 4; ++k) y[q][k] = a.va * x[q][k];
      axpy44(y, a.vb, e);
      store_out<TF32>(a.f2, nullptr, a.hi2, a.lo2, a.fmt, a.so2, i, st, y, xl);
    }
    store_out<TF32>(a.f, a.d, a.hi, a.lo, a.fmt, a.so, i, st, x, xl);
  }
  __syncwarp();
}

// 32 accumulator columns of this lane's row, scaled, into the warp's staging tile
__device__ __forceinline__ void stage_chunk(const float (&v)[32], float inv, int lane, float (*t)[33]) {
#pragma unroll
  for (int i = 0; i < 32; ++i) t[lane][i] = v[i] * inv;
  __syncwarp();
}

template <int BN>
__global__ void __launch_bounds__(192, 1)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap mAhi, const __grid_constant__ CUtensorMap mAlo,
                   const __grid_constant__ CUtensorMap mBhi, const __grid_constant__ CUtensorMap mBlo,
                   const __grid_constant__ CUtensorMap mA2hi, const __grid_constant__ CUtensorMap mA2lo,
                   const __grid_constant__ CUtensorMap mB2hi, const __grid_constant__ CUtensorMap mB2lo, TcArgs a) {
  constexpr int B_BYTES = BN * BK * 2;
  constexpr uint32_t TMEM_COLS = 2 * BN;   // two accumulators: 256 or 512 columns
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STAGES * A_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(sB + STAGES * B_BYTES);
  uint64_t* empty = full + STAGES;
  uint64_t* accf = empty + STAGES;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(accf + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int tm, tn;
  if (a.tile_list) {
    tm = a.tile_list[2 * blockIdx.x];
    tn = a.tile_list[2 * blockIdx.x + 1];
  } else {
    // grouped raster: GROUP_M row panels at a time, so that the CTAs in flight
    // share their A and B panels in L2
    const int tiles_m = a.n / BM;
    const int per_group = kGroupM * a.tiles_n;
    const int g = blockIdx.x / per_group, r = blockIdx.x % per_group;
    const int first = g * kGroupM;
    const int gm = min(tiles_m - first, kGroupM);
    tm = first + r % gm;
    tn = r / gm;
  }
  // a tile outside the matrix (a bad tile list) is reported, never stored
  if (tm < 0 || tm >= a.n / BM || tn < 0 || tn >= a.tiles_n) {
    if (threadIdx.x == 0 && a.err) atomicExch(a.err, 4);
    return;
  }

  if (warp == 0 && lane == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(accf, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  const int nk = a.K / BK;
  const int total = a.nseg * a.pairs * nk;
  bool ok = true;

  if (warp == 0) {
    if (lane == 0) {
      KSeg q;
      kseg_begin(a, nk, q);
      int kb = 0;
      for (; kb < total; ++kb, kseg_next(a, nk, q)) {
        const int s = kb % STAGES;
        const uint32_t ph = (kb / STAGES) & 1;
        if (kb >= STAGES && !mbar_wait_fast(&empty[s], ph ^ 1)) {
          ok = false;
          break;
        }
        mbar_expect_tx(&full[s], A_BYTES + B_BYTES);
        const int kk = q.kidx * BK;
        const CUtensorMap* ma = (q.kind == 2) ? (q.pr ? &mA2lo : &mAlo) : (q.pr ? &mA2hi : &mAhi);
        const CUtensorMap* mb = (q.kind == 1) ? (q.pr ? &mB2lo : &mBlo) : (q.pr ? &mB2hi : &mBhi);
        tma_load_2d(sA + s * A_BYTES, ma, kk, tm * BM, &full[s]);
        tma_load_2d(sB + s * B_BYTES, mb, kk, tn * BN, &full[s]);
      }
      if (!ok) {
        atomicExch(a.err, 1);
        drain_ring(full, STAGES, kb % STAGES, (kb / STAGES) & 1, kb < STAGES);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_f16 = instr_desc(BN, 0);
      constexpr uint32_t idesc_bf16 = instr_desc(BN, 1);
      const uint32_t idesc = a.fmt ? idesc_bf16 : idesc_f16;
      for (int kb = 0; kb < total; ++kb) {
        const int s = kb % STAGES;
        const uint32_t ph = (kb / STAGES) & 1;
        if (!mbar_wait_fast(&full[s], ph)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int nk0 = acc1_start(a, nk);                // first K block of accumulator 1
        const uint32_t dcol = kb >= nk0 ? (uint32_t)BN : 0u;
        const bool first = (kb == 0) || (kb == nk0);
#pragma unroll
        for (int j = 0; j < BK / 16; ++j) {
          const uint64_t ad = smem_desc(sA + s * A_BYTES + j * 32);
          const uint64_t bd = smem_desc(sB + s * B_BYTES + j * 32);
          mma_f16(tmem + dcol, ad, bd, idesc, (first && j == 0) ? 0u : 1u);
        }
        mma_commit(&empty[s]);
      }
      mma_commit(accf);
      if (!ok) atomicExch(a.err, 2);
    }
  } else {
    // epilogue warps 2..5: TMEM lanes 32 * (warp % 4) ..
    const int q = warp & 3;
    prefetch_sides<BN>(a, tm, tn, (warp - 2) * 32 + lane, 128);   // while the tensor cores run
    if (!mbar_wait(accf, 0)) {
      if (lane == 0) atomicExch(a.err, 3);
    } else {
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int row0 = tm * BM + q * 32;
      const EpiRegs er = load_epi(a);
      // per-warp 32 x 33 staging tile in the (now idle) operand ring
      float(*t)[33] = reinterpret_cast<float(*)[33]>(sA + q * (32 * 33 * 4));
      for (int ch = 0; ch < BN / 32; ++ch) {
        float v[32];
        tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(ch * 32), v);
        if (a.nseg > 1 || a.split_acc) {
          float w[32];
          tmem_ld32(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(BN + ch * 32), w);
#pragma unroll
          for (int i = 0; i < 32; ++i) v[i] += w[i];
        }
        if (er.sym && tn * BN + ch * 32 < row0) continue;
        stage_chunk(v, er.inv, lane, t);
        epilogue_chunk<false>(er, row0, tn * BN + ch * 32, lane, t);
      }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// Persistent variant: one CTA per SM walks the tiles id = blockIdx.x, blockIdx.x + gridDim.x, ...
// The producer and MMA threads run ahead into the next tile while the epilogue writes the previous
// one.  A tile's hi*hi sum runs in chunks of chunk_kb K blocks, each accumulated by itself in one of two
// TMEM accumulators that alternate from chunk to chunk (and across tiles); a single product is one
// chunk.  The epilogue warps read each finished chunk (tcgen05.ld), add it to the tile's sum in
// registers (round-to-nearest FP32) and release the accumulator at once, while the other one fills.
// Two column groups of four warps share a tile (BN / 2 sums per thread; one group for BN = 32).
//
// The corrections of a split product (hi*lo, lo*hi, 2^-11 of the whole) have accumulators of their own.
// Tiles of up to 128 columns have TMEM for two more, alternating from tile to tile: each K block's hi
// and lo parts are loaded once (two slots) and all three products taken from them, and the corrections
// are added last.  The ring's turn-around is about 2 us a slot at any width, so a third fewer slots are
// a third less time in the K loop: n = 640 symmetric 14.1 -> 12.0 us, 1408 25.7 -> 21.8, 2048 42.3 -> 37.0.
// Tiles of 256 columns take the corrections as a first chunk, which runs while the epilogue still writes
// the tile before, and load the hi parts a second time.  (One accumulator for all three products had
// three times the error.)
//
// The tensor core truncates as it accumulates, so a sum's error grows with its length; with the sums in
// registers a chunk costs its one tcgen05.ld pass.  (The sums used to live in TMEM, each fold a load, a
// load, an add and a store that the next chunk had to wait for.)  A tcgen05.ld holds up the MMAs
// beside it by a time that hardly depends on its size: with 256-wide tiles and 512-long chunks, n = 8192
// takes 2.46 ms with loads of 32 columns and 2.30 ms with loads of 64.
//
// Barriers: full/empty (operand ring), acc_full[2] (MMA -> epilogue), acc_free[2] (epilogue -> MMA,
// one arrival per epilogue warp).  Chunk c of the CTA uses accumulator c % 2 and waits for release
// c / 2 - 1 of it, so no barrier can run two phases ahead of its waiter.  Every wait is bounded; a
// role that gives up records an error and raises a shared abort flag that ends the other roles' loops.

// Grouped launch (tab != null): tile id -> problem p of the group and its tile lid; tiles_per
// tiles per problem.  Otherwise one problem.
__device__ __forceinline__ void group_tile(const TcEntry* tab, int tiles_per, int id, int& p, int& lid) {
  if (tab) {
    p = id / tiles_per;
    lid = id - p * tiles_per;
  } else {
    p = 0;
    lid = id;
  }
}

// K-block order of one tile (the producer and the MMA thread walk it alike): the Cn correction
// K blocks first (hi*lo, lo*hi of pair 0, then of pair 1), then the hi*hi sequence (pair 0's K
// blocks, then pair 1's).  Counters only, no divisions.
struct KWalk {
  int phase;           // 0: corrections, 1: hi*hi
  int pr, kind, kidx;  // current K block: operand pair, split part (0 hi*hi, 1 hi*lo, 2 lo*hi), index
  int h, c;            // hi*hi and correction K blocks issued before the current one
};

__device__ __forceinline__ void kwalk_begin(KWalk& w, int Cn) {
  w.phase = Cn > 0 ? 0 : 1;
  w.pr = w.kidx = 0;
  w.kind = Cn > 0 ? 1 : 0;
  w.h = w.c = 0;
}

__device__ __forceinline__ void kwalk_next(KWalk& w, int nk, int Cn) {
  if (w.phase == 0) {
    ++w.c;
    if (++w.kidx == nk) {
      w.kidx = 0;
      if (w.kind == 1) {
        w.kind = 2;
      } else {
        w.kind = 1;
        ++w.pr;
      }
    }
    if (w.c == Cn) {
      w.phase = 1;
      w.pr = w.kind = w.kidx = 0;
    }
    return;
  }
  ++w.h;
  if (++w.kidx == nk) {
    w.kidx = 0;
    ++w.pr;
  }
}

// Shape of a persistent CTA with tiles of width BN: epilogue column groups and warps, columns per
// warp, ring stages (as many as fit beside the staging tiles).
template <int BN>
struct PCfg {
  static constexpr int CG = BN >= 64 ? 2 : 1;
  static constexpr int NEPI = 4 * CG;
  static constexpr int THREADS = 128 + 32 * NEPI;   // warpgroup 0: producer and MMA warps (and two idle ones)
  static constexpr int COLS = BN / CG;
  // split products of up to 128 columns load each K block's hi and lo parts once (two slots) and do all
  // three products from them
  static constexpr bool ONCE = BN <= 128;
  static constexpr int STG = BN == 256 ? 4 : BN == 128 ? 6 : BN == 64 ? 8 : 10;   // even where ONCE
  static constexpr uint32_t TMEM_COLS = (ONCE ? 4 : 2) * BN;   // ONCE: two accumulators for corrections
  static constexpr int B_BYTES = BN * BK * 2;
  static constexpr int STAGE_TILE = 32 * 33 * 4;
  static constexpr int SMEM = STG * (A_BYTES + B_BYTES) + NEPI * STAGE_TILE + (2 * STG + 5) * 8 + 16 + 1024;
};

// ---- the two single-thread loops of the persistent kernel: 32-bit shared addresses throughout ----

__device__ __forceinline__ bool bar_spin(uint32_t bar, uint32_t parity) {
  for (int it = 0; it < (kWaitLimit << 4); ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void bar_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// one K block's A and B tiles into a ring slot
__device__ __forceinline__ void load_slot(uint32_t bar, uint32_t bytes, uint32_t da, const CUtensorMap* ma, uint32_t db,
                                          const CUtensorMap* mb, int x, int ya, int yb) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(da),
      "l"(reinterpret_cast<uint64_t>(ma)), "r"(x), "r"(ya), "r"(bar)
      : "memory");
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(db),
      "l"(reinterpret_cast<uint64_t>(mb)), "r"(x), "r"(yb), "r"(bar)
      : "memory");
}

// Shared-memory descriptors (smem_desc) as words: the low one holds the address / 16, the high one is constant.
constexpr uint32_t kDescHi = (1024u >> 4) | (1u << 14) | (2u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return (addr >> 4) | (1u << 16); }

template <bool TF32>
__device__ __forceinline__ void mma_words(uint32_t d, uint32_t alo, uint32_t blo, uint32_t idesc, uint32_t accumulate) {
  if constexpr (TF32)
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], da, db, %4, p;\n\t}" ::"r"(d),
        "r"(alo), "r"(blo), "r"(kDescHi), "r"(idesc), "r"(accumulate)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b64 da, db;\n\t"
        "setp.ne.b32 p, %5, 0;\n\t"
        "mov.b64 da, {%1, %3};\n\tmov.b64 db, {%2, %3};\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %4, p;\n\t}" ::"r"(d),
        "r"(alo), "r"(blo), "r"(kDescHi), "r"(idesc), "r"(accumulate)
        : "memory");
}

// TF32: operands are TF32 words (kind::tf32, 32-element K blocks); else FP16 or BF16 by a.fmt.
template <int BN, bool TF32>
__global__ void __launch_bounds__(PCfg<BN>::THREADS, 1)
    gemm_tc_persistent_kernel(const __grid_constant__ CUtensorMap mAhi, const __grid_constant__ CUtensorMap mAlo,
                              const __grid_constant__ CUtensorMap mBhi, const __grid_constant__ CUtensorMap mBlo,
                              const __grid_constant__ CUtensorMap mA2hi, const __grid_constant__ CUtensorMap mA2lo,
                              const __grid_constant__ CUtensorMap mB2hi, const __grid_constant__ CUtensorMap mB2lo,
                              TcArgs a, int ntiles, const TcEntry* tab, int tiles_per) {
  using Cfg = PCfg<BN>;
  constexpr int STG = Cfg::STG, B_BYTES = Cfg::B_BYTES, COLS = Cfg::COLS;
  constexpr uint32_t TMEM_COLS = Cfg::TMEM_COLS;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + STG * A_BYTES;
  uint8_t* stage = sB + STG * B_BYTES;     // one staging tile per epilogue warp
  uint64_t* full = reinterpret_cast<uint64_t*>(stage + Cfg::NEPI * Cfg::STAGE_TILE);
  uint64_t* empty = full + STG;
  uint64_t* acc_full = empty + STG;        // [2]
  uint64_t* acc_free = acc_full + 2;       // [2]
  uint64_t* drain = acc_full + 4;          // completion of the last MMAs after a wait that gave up
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp == 0 && lane == 0) {
    for (int s = 0; s < STG; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full[0], 1);
    mbar_init(&acc_full[1], 1);
    mbar_init(&acc_free[0], Cfg::NEPI);
    mbar_init(&acc_free[1], Cfg::NEPI);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  grid_wait();   // the prologue above overlaps the kernel before
  constexpr int bk = TF32 ? BK / 2 : BK;           // elements per K block (one 128-byte row)
  const int nk = a.K / bk;
  const bool once = Cfg::ONCE && a.nseg > 1;
  const int H = a.pairs * nk;                      // hi*hi K blocks
  const int Cn = once ? 0 : (a.nseg - 1) * H;      // correction K blocks in a chunk of their own (the first)
  const int total = Cn + H;
  const int Lc = (a.nseg > 1 && a.chunk_kb > 0 && a.chunk_kb < H) ? a.chunk_kb : H;   // hi*hi chunk
  const int nch = (Cn > 0 ? 1 : 0) + (H + Lc - 1) / Lc;                               // chunks per tile

  // BN = 256 holds 128 sums a thread: the 384 threads are launched with 168 registers each, 64,512 in
  // all; the producer's warpgroup keeps 40 a thread (128 x 40) and the epilogue's two get 232 (256 x 232)
  if (warp < 4) {
    if constexpr (BN == 256) asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
    const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB), full0 = smem_u32(full), empty0 = smem_u32(empty);
    uint32_t slot = 0, ph = 0;         // ring slot and the parity of its current use
    bool ok = true;
    if (warp == 0 && lane == 0) {
      bool first = true;               // the ring's first use needs no release
      int last_p = -1;
      for (int id = blockIdx.x; id < ntiles && ok && !*abort_flag; id += gridDim.x) {
        int tm, tn, p, lid;
        group_tile(tab, tiles_per, id, p, lid);
        if (!tile_coords(a, lid, tm, tn)) {
          atomicExch(a.err, 4);
          *abort_flag = 1;
          break;
        }
        const CUtensorMap* maps = tab ? tab[p].map : nullptr;   // grouped: this problem's maps
        if (maps && p != last_p) {
          for (int i = 0; i < 8; ++i) tensormap_acquire(&maps[i]);
          last_p = p;
        }
        // Segments of K blocks, two loads of A and B tiles per K block in the first kind:
        //   once    the hi parts, the lo parts
        //   else    corrections: A hi and B lo, A lo and B hi; then (kind 1) the hi parts alone
        // each for the pair and, in pair products, the swapped pair.
        for (int sg = (a.nseg > 1 ? 0 : a.pairs); sg < (once ? 1 : 2) * a.pairs && ok; ++sg) {
          const int pr = sg % a.pairs;
          const bool two = sg < a.pairs;
          const CUtensorMap* ahi = maps ? &maps[pr ? 4 : 0] : pr ? &mA2hi : &mAhi;
          const CUtensorMap* alo_ = maps ? &maps[pr ? 5 : 1] : pr ? &mA2lo : &mAlo;
          const CUtensorMap* bhi = maps ? &maps[pr ? 6 : 2] : pr ? &mB2hi : &mBhi;
          const CUtensorMap* blo_ = maps ? &maps[pr ? 7 : 3] : pr ? &mB2lo : &mBlo;
          auto put = [&](const CUtensorMap* ma, const CUtensorMap* mb, int k) -> bool {
            if (!first && !bar_spin(empty0 + 8 * slot, ph ^ 1)) {
              atomicExch(a.err, 1);
              *abort_flag = 1;
              return false;
            }
            load_slot(full0 + 8 * slot, A_BYTES + B_BYTES, a0 + slot * A_BYTES, ma, b0 + slot * B_BYTES, mb, k, tm * BM,
                      tn * BN);
            if (++slot == STG) {
              slot = 0;
              ph ^= 1;
              first = false;
            }
            return true;
          };
          if (two) {
            const CUtensorMap* b1 = once ? bhi : blo_;
            const CUtensorMap* b2 = once ? blo_ : bhi;
            for (int k = 0; k < a.K && ok; k += bk) ok = put(ahi, b1, k) && put(alo_, b2, k);
          } else {
            for (int k = 0; k < a.K && ok; k += bk) ok = put(ahi, bhi, k);
          }
        }
      }
      if (*abort_flag) drain_ring(full, STG, slot, ph, first);
    } else if (warp == 1 && lane == 0) {
      constexpr uint32_t idesc_f16 = instr_desc(BN, 0);
      constexpr uint32_t idesc_bf16 = instr_desc(BN, 1);
      constexpr uint32_t idesc_tf32 = instr_desc(BN, 2);
      const uint32_t idesc = TF32 ? idesc_tf32 : a.fmt ? idesc_bf16 : idesc_f16;
      const uint32_t alo0 = desc_lo(a0), blo0 = desc_lo(b0);
      const uint32_t accf0 = smem_u32(acc_full), accr0 = smem_u32(acc_free);
      uint32_t alo = alo0, blo = blo0, c = 0;   // descriptors of the slot; chunks of this CTA so far
      uint32_t par = 0;                // once: the tile's correction accumulator
      for (int id = blockIdx.x; id < ntiles && ok && !*abort_flag; id += gridDim.x, par ^= 1) {
        int tm, tn, p, lid;
        group_tile(tab, tiles_per, id, p, lid);
        if (!tile_coords(a, lid, tm, tn)) break;
        int done = 0;                  // K blocks of this tile so far
        for (int ch = 0; ch < nch && ok; ++ch, ++c) {
          const uint32_t b = c & 1;
          if (c >= 2) {                // the epilogue has read this accumulator's previous chunk
            if (!bar_spin(accr0 + 8 * b, ((c >> 1) - 1) & 1) || *abort_flag) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          const int len = (ch == 0 && Cn > 0) ? Cn : min(Lc, total - done);
          done += len;
          const uint32_t d = tmem + b * BN;
          uint32_t acc = 0;
          for (int i = 0; i < len; ++i) {
            if (!bar_spin(full0 + 8 * slot, ph)) {
              ok = false;
              break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            mma_words<TF32>(d, alo, blo, idesc, acc);
            mma_words<TF32>(d, alo + 2, blo + 2, idesc, 1u);
            mma_words<TF32>(d, alo + 4, blo + 4, idesc, 1u);
            mma_words<TF32>(d, alo + 6, blo + 6, idesc, 1u);
            acc = 1;
            if (once) {                // the lo slot is the next one of the same round (STG is even)
              if (!bar_spin(full0 + 8 * slot + 8, ph)) {
                ok = false;
                break;
              }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
              const uint32_t dc = tmem + (2 + par) * BN;
              const uint32_t al = alo + (A_BYTES >> 4), bl = blo + (B_BYTES >> 4);
              const uint32_t fc = (ch == 0 && i == 0) ? 0u : 1u;
#pragma unroll
              for (int j = 0; j < 4; ++j) mma_words<TF32>(dc, alo + 2 * j, bl + 2 * j, idesc, j == 0 ? fc : 1u);
#pragma unroll
              for (int j = 0; j < 4; ++j) mma_words<TF32>(dc, al + 2 * j, blo + 2 * j, idesc, 1u);
              bar_commit(empty0 + 8 * slot);
              ++slot;
              alo = al;
              blo = bl;
            }
            bar_commit(empty0 + 8 * slot);
            alo += A_BYTES >> 4;
            blo += B_BYTES >> 4;
            if (++slot == STG) {
              slot = 0;
              ph ^= 1;
              alo = alo0;
              blo = blo0;
            }
          }
          if (ok) bar_commit(accf0 + 8 * b);
        }
        if (!ok) {
          atomicExch(a.err, 2);
          *abort_flag = 1;
        }
      }
      if (*abort_flag) {
        bar_commit(smem_u32(drain));
        mbar_wait(drain, 0);
      }
    }
  } else {
    if constexpr (BN == 256) asm volatile("setmaxnreg.inc.sync.aligned.u32 232;");
    // epilogue warps: TMEM lanes 32 * (warp % 4) .., columns COLS * cg ..
    const int q = warp & 3, cg = (warp - 4) >> 2;
    float(*t)[33] = reinterpret_cast<float(*)[33]>(stage + (warp - 4) * Cfg::STAGE_TILE);
    const uint32_t tbase = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(cg * COLS);
    uint32_t c = 0, par = 0;
    for (int id = blockIdx.x; id < ntiles && !*abort_flag; id += gridDim.x, par ^= 1) {
      int tm, tn, p, lid;
      group_tile(tab, tiles_per, id, p, lid);
      if (!tile_coords(a, lid, tm, tn)) break;
      EpiRegs er;                      // this problem's epilogue
      if (tab)
        er = load_epi(tab[p].args);
      else
        er = load_epi(a);
      prefetch_sides<BN>(er, tm, tn, (warp - 4) * 32 + lane, 32 * Cfg::NEPI);
      float sum[COLS / 32][32];
      bool ok = true;
      for (int ch = 0; ch < nch; ++ch, ++c) {
        const int b = c & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[b], (c >> 1) & 1));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if constexpr (COLS == 128) {
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            uint32_t v[64];
            tmem_ld64_nowait(tbase + (uint32_t)(b * BN + x * 64), v);
            tmem_wait_ld64(v);
#pragma unroll
            for (int i = 0; i < 64; ++i) {
              float& y = sum[2 * x + i / 32][i % 32];
              y = ch ? y + __uint_as_float(v[i]) : __uint_as_float(v[i]);
            }
          }
        } else {
#pragma unroll
          for (int x = 0; x < COLS / 32; ++x) {
            float v[32];
            tmem_ld32(tbase + (uint32_t)(b * BN + x * 32), v);
#pragma unroll
            for (int i = 0; i < 32; ++i) sum[x][i] = ch ? sum[x][i] + v[i] : v[i];
          }
          if (once && ch == nch - 1) {   // the tile's corrections
#pragma unroll
            for (int x = 0; x < COLS / 32; ++x) {
              float v[32];
              tmem_ld32(tbase + (uint32_t)((2 + par) * BN + x * 32), v);
#pragma unroll
              for (int i = 0; i < 32; ++i) sum[x][i] += v[i];
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_free[b]);
      }
      if (!ok || *abort_flag) {
        if (lane == 0) atomicExch(a.err, 3);
        *abort_flag = 1;
        break;
      }
      const int row0 = tm * BM + q * 32, colw = tn * BN + cg * COLS;
#pragma unroll 1
      for (int x = 0; x < COLS / 32; ++x) {   // one copy of the epilogue's code; the sums' index stays static
        if (er.sym && colw + x * 32 < row0) continue;
#pragma unroll
        for (int y = 0; y < COLS / 32; ++y)
          if (y == x) stage_chunk(sum[y], er.inv, lane, t);
        epilogue_chunk<TF32>(er, row0, colw + x * 32, lane, t);
      }
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---- two-SM products (cta_group::2) ----
//
// A cluster of two CTAs on two SMs computes a 256 x 256 output tile with tcgen05.mma.cta_group::2
// (M = 256, N = 256, K = 16): CTA r of the pair holds rows 128 r .. 128 r + 127 of the A tile and
// of the B tile in its own shared memory and rows 128 r .. of the accumulator in its own TMEM.
// The tensor cores of both SMs read both CTAs' operands, so each SM stages half as many B bytes
// per flop as the one-SM product: 32 KB per 64-wide K block instead of 48 KB, six ring stages
// instead of four, a third less shared-memory traffic per flop.  Single products alternate
// accumulators from tile to tile.  Split products start from the corrections and fold 1024-long
// chunks of hi*hi into them through TMEM, by both CTAs' epilogue warps on their own TMEM lanes: another
// order of sums than the one-SM kernel's (512-long chunks in registers), so the two agree to the error
// bound of a product and not to the bit.
//
// Roles.  Both CTAs: warp 0 lane 0 loads the CTA's A and B halves of each K block by TMA,
// signalling the leader CTA's (rank 0) full barrier; warps 2-5 run the epilogue.  Leader only:
// warp 1 lane 0 waits for both halves (full), issues the MMAs and commits to the empty, acc_full
// barriers of both CTAs (multicast).  The epilogue warps of both CTAs release accumulators on the
// leader's acc_free barriers (eight warp arrivals per phase, four of them remote).  TMEM is
// allocated and freed collectively by warp 1 of both CTAs.  Cluster barriers after the barrier
// set-up and before the TMEM release are reached by every thread of both CTAs; every other wait
// is bounded.
constexpr int PSTAGES = 6;
constexpr int PB_BYTES = 128 * BK * 2;           // a CTA's half of the 256-row B tile
constexpr int kPairGroupM = 8;                   // 256-row panels per raster group
constexpr int kPairChunkKb = 16;                 // hi*hi chunk (its folds go through TMEM)

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// the shared::cluster address of the same shared-memory word in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_to_rank(const void* p, uint32_t rank) {
  uint32_t out;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(out) : "r"(smem_u32(p)), "r"(rank));
  return out;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}

// TMA load into this CTA's shared memory that signals an mbarrier of either CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(void* dst, const CUtensorMap* map, int x, int y, uint32_t bar_cluster) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster)
      : "memory");
}

__device__ __forceinline__ void mma_f16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// arrive on the same barrier in both CTAs of the pair once the MMAs issued so far complete
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((unsigned short)3)
      : "memory");
}

// arrive on this CTA's barrier once the pair MMAs issued so far complete
__device__ __forceinline__ void mma_commit_pair_local(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ bool pair_tile_coords(const TcArgs& a, int id, int& tm, int& tn) {
  const int tiles = a.n / 256;
  if (a.tile_list) {
    tm = a.tile_list[2 * id];
    tn = a.tile_list[2 * id + 1];
  } else {
    const int per_group = kPairGroupM * tiles;
    const int g = id / per_group, r = id % per_group;
    const int first = g * kPairGroupM;
    const int gm = min(tiles - first, kPairGroupM);
    tm = first + r % gm;
    tn = r / gm;
  }
  return tm >= 0 && tm < tiles && tn >= 0 && tn < tiles;
}

__global__ void __launch_bounds__(192, 1)
    gemm_tc_pair_kernel(const __grid_constant__ CUtensorMap mAhi, const __grid_constant__ CUtensorMap mAlo,
                        const __grid_constant__ CUtensorMap mBhi, const __grid_constant__ CUtensorMap mBlo,
                        const __grid_constant__ CUtensorMap mA2hi, const __grid_constant__ CUtensorMap mA2lo,
                        const __grid_constant__ CUtensorMap mB2hi, const __grid_constant__ CUtensorMap mB2lo,
                        TcArgs a, int ntiles) {
  constexpr int BN = 256;
  constexpr uint32_t TMEM_COLS = 2 * BN;
  constexpr int STAGE_TILE = 32 * 33 * 4;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + PSTAGES * A_BYTES;
  uint8_t* stage = sB + PSTAGES * PB_BYTES;
  uint64_t* full = reinterpret_cast<uint64_t*>(stage + 4 * STAGE_TILE);
  uint64_t* empty = full + PSTAGES;
  uint64_t* acc_full = empty + PSTAGES;    // [2]
  uint64_t* acc_free = acc_full + 2;       // [2], used in the leader
  uint64_t* drain = acc_full + 4;          // leader: completion of the last MMAs before teardown
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = (rank == 0);
  const int pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;
  if (warp == 0 && lane == 0) {
    for (int s = 0; s < PSTAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(&acc_full[0], 1);
    mbar_init(&acc_full[1], 1);
    mbar_init(&acc_free[0], 8);
    mbar_init(&acc_free[1], 8);
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();   // both CTAs' barriers exist before any remote signal
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  const int nk = a.K / BK;
  const int total = a.nseg * a.pairs * nk;
  const bool chunked = a.nseg > 1;
  const int H = a.pairs * nk;
  const int Cn = total - H;
  const int Lc = (chunked && a.chunk_kb > 0 && a.chunk_kb < H) ? a.chunk_kb : H;
  const int nchunks = (H + Lc - 1) / Lc;
  const int nfold = chunked ? nchunks : 0;

  if (warp == 0) {
    if (lane == 0) {
      const uint32_t full_leader0 = map_to_rank(&full[0], 0);   // leader's full[0]; stages 8 bytes apart
      uint32_t g = 0;
      bool ok = true;
      for (int id = pair; id < ntiles && ok && !*abort_flag; id += npairs) {
        int tm, tn;
        if (!pair_tile_coords(a, id, tm, tn)) {
          atomicExch(a.err, 4);
          *abort_flag = 1;
          break;
        }
        const int arow = tm * 256 + (int)rank * 128, brow = tn * 256 + (int)rank * 128;
        KWalk w;
        kwalk_begin(w, Cn);
        for (int kb = 0; kb < total; ++kb, ++g, kwalk_next(w, nk, Cn)) {
          const int s = g % PSTAGES;
          const uint32_t ph = (g / PSTAGES) & 1;
          if (g >= PSTAGES && !mbar_wait_fast(&empty[s], ph ^ 1)) {
            atomicExch(a.err, 1);
            *abort_flag = 1;
            ok = false;
            break;
          }
          if (leader) mbar_expect_tx(&full[s], 2 * (A_BYTES + PB_BYTES));   // both CTAs' halves
          const int kk = w.kidx * BK;
          const CUtensorMap* ma = (w.kind == 2) ? (w.pr ? &mA2lo : &mAlo) : (w.pr ? &mA2hi : &mAhi);
          const CUtensorMap* mb = (w.kind == 1) ? (w.pr ? &mB2lo : &mBlo) : (w.pr ? &mB2hi : &mBhi);
          const uint32_t bar = full_leader0 + 8u * (uint32_t)s;
          tma_load_2d_pair(sA + s * A_BYTES, ma, kk, arow, bar);
          tma_load_2d_pair(sB + s * PB_BYTES, mb, kk, brow, bar);
        }
      }
      // both CTAs' copies signal the leader's barriers
      if (leader && *abort_flag) drain_ring(full, PSTAGES, g % PSTAGES, (g / PSTAGES) & 1, g < PSTAGES);
    }
  } else if (warp == 1) {
    if (lane == 0 && leader) {
      constexpr uint32_t idesc_f16 = instr_desc_m(256, BN, 0);
      constexpr uint32_t idesc_bf16 = instr_desc_m(256, BN, 1);
      const uint32_t idesc = a.fmt ? idesc_bf16 : idesc_f16;
      uint32_t g = 0;
      int it = 0;
      int uses0 = 0, uses1 = 0;
      int par = 0;
      bool issued = false;
      for (int id = pair; id < ntiles && !*abort_flag; id += npairs, ++it, par ^= 1) {
        int tm, tn;
        if (!pair_tile_coords(a, id, tm, tn)) break;
        bool ok = true;
        const int buf = it & 1;
        int cur = 0;
        int bnd = 0;
        KWalk w;
        kwalk_begin(w, Cn);
        for (int kb = 0; kb < total; ++kb, ++g, kwalk_next(w, nk, Cn)) {
          int fresh = -1;
          if (!chunked) {
            if (kb == 0) fresh = buf;
          } else if (w.phase == 0) {
            if (w.c == 0) fresh = par;                     // corrections: the tile's sum accumulator
          } else if (w.h == bnd) {
            if (bnd > 0) mma_commit_pair(&acc_full[0]);
            fresh = par ^ 1;                               // next hi*hi chunk
            bnd += Lc;
          }
          if (fresh >= 0) {
            const int u = chunked ? (fresh ? uses1 : uses0) : (it >> 1);
            if (u > 0) {
              if (!mbar_wait_fast(&acc_free[fresh], (uint32_t)((u - 1) & 1)) || *abort_flag) {
                ok = false;
                break;
              }
              asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            }
            if (chunked) {
              if (fresh)
                ++uses1;
              else
                ++uses0;
            }
            cur = fresh;
          }
          const int s = g % PSTAGES;
          const uint32_t ph = (g / PSTAGES) & 1;
          if (!mbar_wait_fast(&full[s], ph)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t dcol = cur ? (uint32_t)BN : 0u;
#pragma unroll
          for (int j = 0; j < BK / 16; ++j) {
            const uint64_t ad = smem_desc(sA + s * A_BYTES + j * 32);
            const uint64_t bd = smem_desc(sB + s * PB_BYTES + j * 32);
            mma_f16_pair(tmem + dcol, ad, bd, idesc, (fresh >= 0 && j == 0) ? 0u : 1u);
          }
          issued = true;
          mma_commit_pair(&empty[s]);
        }
        if (!ok) {
          atomicExch(a.err, 2);
          *abort_flag = 1;
          break;
        }
        mma_commit_pair(&acc_full[chunked ? 0 : buf]);
      }
      // no MMA may still write either CTA's TMEM when the pair frees it
      if (issued) {
        mma_commit_pair_local(drain);
        if (!mbar_wait(drain, 0)) atomicExch(a.err, 5);
      }
    }
  } else {
    const int q = warp & 3;
    float(*t)[33] = reinterpret_cast<float(*)[33]>(stage + q * STAGE_TILE);
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const EpiRegs er = load_epi(a);
    const uint32_t free_leader0 = map_to_rank(&acc_free[0], 0), free_leader1 = map_to_rank(&acc_free[1], 0);
    int it = 0;
    uint32_t ev = 0;
    int par = 0;
    for (int id = pair; id < ntiles && !*abort_flag; id += npairs, ++it, par ^= 1) {
      int tm, tn;
      if (!pair_tile_coords(a, id, tm, tn)) break;
      const int tm128 = 2 * tm + (int)rank;          // this CTA's 128-row panel
      prefetch_sides<BN>(a, tm128, tn, (warp - 2) * 32 + lane, 128);
      int src;
      bool ok = true;
      if (!chunked) {
        src = it & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[src], (uint32_t)((it >> 1) & 1)));
        if (ok) asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      } else {
        src = par;
        for (int f = 1; f <= nfold && ok; ++f, ++ev) {
          ok = __all_sync(0xffffffffu, mbar_wait(&acc_full[0], ev & 1));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int dst = par, from = par ^ 1;
          for (int ch = 0; ch < BN / 64; ++ch) {
            uint32_t v[64], u[64];
            tmem_ld64_nowait(tmem + lane_base + (uint32_t)(from * BN + ch * 64), v);
            tmem_ld64_nowait(tmem + lane_base + (uint32_t)(dst * BN + ch * 64), u);
            tmem_wait_ld64(v);
            tmem_after_wait64(u);
#pragma unroll
            for (int i = 0; i < 64; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(u[i]));
            tmem_st64(tmem + lane_base + (uint32_t)(dst * BN + ch * 64), v);
          }
          asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(from ? free_leader1 : free_leader0);
          src = dst;
        }
      }
      if (!ok || *abort_flag) {
        if (lane == 0) atomicExch(a.err, 3);
        *abort_flag = 1;
        break;
      }
      const int row0 = tm128 * BM + q * 32;
      for (int ch = 0; ch < BN / 32; ++ch) {
        float v[32];
        tmem_ld32(tmem + lane_base + (uint32_t)(src * BN + ch * 32), v);
        if (er.sym && tn * BN + ch * 32 < row0) continue;
        stage_chunk(v, er.inv, lane, t);
        epilogue_chunk<false>(er, row0, tn * BN + ch * 32, lane, t);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(src ? free_leader1 : free_leader0);
    }
  }

  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  cluster_sync();   // the peer is done with this CTA's shared memory and TMEM
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// ---- host side: tensor maps ----

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  });
  return fn;
}

struct MapKey {
  const void* p;
  int rows, box, fmt;
  bool operator==(const MapKey& o) const { return p == o.p && rows == o.rows && box == o.box && fmt == o.fmt; }
};
struct MapHash {
  size_t operator()(const MapKey& k) const {
    return std::hash<const void*>()(k.p) ^ (size_t)k.rows * 1315423911u ^ (size_t)k.box * 2654435761u ^ k.fmt;
  }
};

std::mutex g_map_mu;
std::unordered_map<MapKey, CUtensorMap, MapHash> g_maps;

// n x n row-major operand, boxes of one 128-byte swizzle row (64 16-bit or 32 TF32 elements) by
// box_rows rows; fmt 0 FP16, 1 BF16, 2 TF32 (FP32 words)
bool make_map(CUtensorMap* out, const void* base, int n, int box_rows, int fmt) {
  std::lock_guard<std::mutex> lk(g_map_mu);
  MapKey k{base, n, box_rows, fmt};
  auto it = g_maps.find(k);
  if (it != g_maps.end()) {
    *out = it->second;
    return true;
  }
  EncodeTiledFn enc = get_encode();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)n, (cuuint64_t)n};
  const int esz = fmt == 2 ? 4 : 2;
  cuuint64_t strides[1] = {(cuuint64_t)n * esz};
  cuuint32_t box[2] = {(cuuint32_t)(128 / esz), (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUtensorMap m;
  const CUtensorMapDataType dt = fmt == 2   ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                 : fmt == 1 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                            : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  CUresult r = enc(&m, dt, 2,
                   const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                   CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return false;
  g_maps[k] = m;
  *out = m;
  return true;
}

template <int BN>
int smem_bytes() {
  return STAGES * (A_BYTES + BN * BK * 2) + (2 * STAGES + 1) * 8 + 16 + 1024;
}

int smem_bytes_pair() {
  return PSTAGES * (A_BYTES + PB_BYTES) + 4 * 32 * 33 * 4 + (2 * PSTAGES + 5) * 8 + 16 + 1024;
}

// 1: one-SM persistent CTAs (default); 2: two-SM products where n is a multiple of 256
// (XLBOMD_GEMM=pair), else one-SM persistent CTAs; 0: one CTA per output tile
// (XLBOMD_GEMM=classic).
int tc_variant() {
  static int v = -1;
  static std::once_flag once;
  std::call_once(once, [] {
    const char* e = std::getenv("XLBOMD_GEMM");
    const std::string x = e ? std::string(e) : std::string();
    v = (x == "classic") ? 0 : (x == "pair") ? 2 : 1;
  });
  return v;
}

// Per-device launch state: the SM count and whether each kernel's dynamic shared-memory limit
// has been raised on that device (a process may drive several devices).
constexpr int kMaxDevices = 64;
struct DeviceState {
  int sms = 0;
  int pair_clusters = 0;   // co-resident clusters of the two-SM product kernel
  bool smem_set[11] = {};   // 0-3 persistent kernel per width, 4-7 its TF32 form, 8, 9 one-CTA-per-tile, 10 two-SM
};
std::mutex g_dev_mu;
DeviceState g_dev[kMaxDevices];

int current_device() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) dev = 0;
  return dev;
}

int sm_count() {
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(g_dev_mu);
  DeviceState& d = g_dev[dev];
  if (d.sms <= 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      return 148;
    }
    d.sms = n;
  }
  return d.sms;
}

// How many two-SM clusters of the pair kernel fit on the current device at once (its shared
// memory allows one CTA per SM; pairs must sit on SM pairs of one GPC).
int pair_clusters(int smem) {
  const int dev = current_device();
  {
    std::lock_guard<std::mutex> lk(g_dev_mu);
    if (g_dev[dev].pair_clusters > 0) return g_dev[dev].pair_clusters;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2, 1, 1);
  cfg.blockDim = dim3(192, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, gemm_tc_pair_kernel, &cfg) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    n = sm_count() / 2;
  }
  std::lock_guard<std::mutex> lk(g_dev_mu);
  g_dev[dev].pair_clusters = n;
  return n;
}

// Raise kernel `slot`'s dynamic shared-memory limit to `bytes` on the current device (once per
// device; a failed attempt is retried on the next launch).
template <typename Kern>
cudaError_t ensure_smem(int slot, Kern kern, int bytes) {
  const int dev = current_device();
  std::lock_guard<std::mutex> lk(g_dev_mu);
  if (g_dev[dev].smem_set[slot]) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) g_dev[dev].smem_set[slot] = true;
  return e;
}

// Persistent launch with tiles of width BN (grid CTAs, one per SM); TF32 operands (a.fmt = 2)
// take their own instantiation, so the FP16/BF16 kernel keeps compile-time K blocks.
template <int BN>
cudaError_t launch_width(cudaStream_t s, int slot, int grid, const CUtensorMap (&m)[8], const TcArgs& a, int ntiles,
                         const TcEntry* tab, int tiles_per) {
  constexpr int sb = PCfg<BN>::SMEM;
  const bool tf32 = a.fmt == 2;
  auto kern = tf32 ? gemm_tc_persistent_kernel<BN, true> : gemm_tc_persistent_kernel<BN, false>;
  const cudaError_t attr = ensure_smem(slot + (tf32 ? 4 : 0), kern, sb);
  if (attr != cudaSuccess) return attr;
  return launch_chained(s, grid, PCfg<BN>::THREADS, sb, kern, m[0], m[1], m[2], m[3], m[4], m[5], m[6], m[7], a, ntiles,
                        tab, tiles_per);
}

cudaError_t launch_persistent(cudaStream_t s, int width, const CUtensorMap (&m)[8], const TcArgs& a, int ntiles,
                              const TcEntry* tab, int tiles_per) {
  const int grid = std::min(ntiles, sm_count());
  switch (width) {
    case 0: return launch_width<32>(s, 0, grid, m, a, ntiles, tab, tiles_per);
    case 1: return launch_width<64>(s, 1, grid, m, a, ntiles, tab, tiles_per);
    case 2: return launch_width<128>(s, 2, grid, m, a, ntiles, tab, tiles_per);
    default: return launch_width<256>(s, 3, grid, m, a, ntiles, tab, tiles_per);
  }
}

int tiles_of(int n, int width, bool sym, const TcTiles& t) {
  return sym ? t.nsym[width] : (n / BM) * (n / tc_width(width));
}

// Tile width of a persistent launch over nprob problems of size n: 256 where n > 3072 allows it, else the one
// of 32, 64 and 128 with the least waves of tiles times the time of a tile.  (The 256-wide tiles add up
// their corrections apart from the rest, so their results differ from the others' in rounding; a size
// always takes one kind, whatever the number of problems.)  The times of a 128 x w tile relative to
// w = 128 hardly depend on n: a CTA's K loop is bound by the ring's turn-around, about 2 us at any width.
// Above 3072 every second padded size (no multiple of 256) takes 128-wide tiles.  That costs little: dense
// split products in TFLOP/s of 16-bit work, 128-wide n = 3200, 4992, 6272, 8064: 1078, 1297, 1394, 1410;
// 256-wide 3328, 5120, 6400, 8192: 1014, 1289, 1350, 1461 (fewer and larger tiles, an emptier last wave).
int pick_width(int n, int nprob, const TcArgs& a, const TcTiles& t) {
  static const int cost[kTcWidths] = {68, 75, 100, 150};
  if (n > kOnceMaxN && n % 256 == 0) return 3;
  const int sms = sm_count();
  int best = 2;
  long long least = -1;
  for (int w = 0; w < 3; ++w) {
    const long long tiles = (long long)nprob * tiles_of(n, w, a.sym != 0, t);
    const long long c = (tiles + sms - 1) / sms * cost[w];
    if (least < 0 || c < least) {
      least = c;
      best = w;
    }
  }
  return best;
}

}  // namespace

void tc_forget_maps(const void* base) {
  std::lock_guard<std::mutex> lk(g_map_mu);
  for (auto it = g_maps.begin(); it != g_maps.end();) {
    if (it->first.p == base)
      it = g_maps.erase(it);
    else
      ++it;
  }
}

namespace {

// the second pair of p: its own, or the first one swapped
void second_pair(const TcProblem& p, const void* (&q)[4]) {
  const void* own[4] = {p.A2hi, p.A2lo ? p.A2lo : p.A2hi, p.B2hi, p.B2lo ? p.B2lo : p.B2hi};
  const void* swapped[4] = {p.Bhi, p.Blo ? p.Blo : p.Bhi, p.Ahi, p.Alo ? p.Alo : p.Ahi};
  for (int i = 0; i < 4; ++i) q[i] = p.A2hi ? own[i] : swapped[i];
}

}  // namespace

cudaError_t gemm_tc(cudaStream_t s, int n, const TcProblem& prob, const TcTiles& tiles) {
  TcArgs args = prob.epi;
  const void *Ahi = prob.Ahi, *Alo = prob.Alo, *Bhi = prob.Bhi, *Blo = prob.Blo;
  if (n % 128 != 0 || n <= 0) return cudaErrorInvalidValue;
  if (args.pairs != 1 && args.pairs != 2) return cudaErrorInvalidValue;
  const bool wide = (n % 256 == 0);
  if (args.fmt < 0 || args.fmt > 2) return cudaErrorInvalidValue;
  // TF32 operands run on the persistent kernel only
  const int variant = args.fmt == 2 ? 1 : tc_variant();
  const bool two_sm = (variant == 2) && wide && tiles.pair != nullptr;
  const int width = variant == 0 ? (wide ? 3 : 2) : pick_width(n, 1, args, tiles);
  // B boxes: a CTA's 128-row half of the 256-row tile (two-SM), else the tile's bn rows
  const int bn = tc_width(width);
  const int bbox = two_sm ? 128 : bn;
  CUtensorMap mAhi, mAlo, mBhi, mBlo, mA2hi, mA2lo, mB2hi, mB2lo;
  if (!make_map(&mAhi, Ahi, n, BM, args.fmt) || !make_map(&mAlo, Alo ? Alo : Ahi, n, BM, args.fmt) ||
      !make_map(&mBhi, Bhi, n, bbox, args.fmt) || !make_map(&mBlo, Blo ? Blo : Bhi, n, bbox, args.fmt))
    return cudaErrorInvalidValue;
  if (args.pairs == 2) {
    const void* q[4];
    second_pair(prob, q);
    if (!make_map(&mA2hi, q[0], n, BM, args.fmt) || !make_map(&mA2lo, q[1], n, BM, args.fmt) ||
        !make_map(&mB2hi, q[2], n, bbox, args.fmt) || !make_map(&mB2lo, q[3], n, bbox, args.fmt))
      return cudaErrorInvalidValue;
  } else {
    mA2hi = mAhi;
    mA2lo = mAlo;
    mB2hi = mBhi;
    mB2lo = mBlo;
  }
  args.n = n;
  args.K = n;
  if (args.split_acc && n / BK < 2) return cudaErrorInvalidValue;   // both accumulators get K blocks
  args.tiles_n = n / bn;
  if (two_sm) {
    args.chunk_kb = kPairChunkKb;
    int ntiles;
    if (args.sym) {
      args.tile_list = tiles.pair;
      ntiles = tiles.npair;
    } else {
      args.tile_list = nullptr;
      ntiles = (n / 256) * (n / 256);
    }
    const int sb = smem_bytes_pair();
    const cudaError_t attr = ensure_smem(10, gemm_tc_pair_kernel, sb);
    if (attr != cudaSuccess) return attr;
    const int npairs = std::min(ntiles, pair_clusters(sb));
    if (const char* dbg = std::getenv("XLBOMD_DEBUG"))
      if (dbg[0] && dbg[0] != '0')
        std::fprintf(stderr, "[xlbomd] two-SM product n %d: %d tiles on %d CTA pairs (%d co-resident)\n", n, ntiles,
                     npairs, pair_clusters(sb));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * npairs, 1, 1);
    cfg.blockDim = dim3(192, 1, 1);
    cfg.dynamicSmemBytes = sb;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, gemm_tc_pair_kernel, mAhi, mAlo, mBhi, mBlo, mA2hi, mA2lo, mB2hi,
                                             mB2lo, args, ntiles);
    note_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
  }
  args.tile_list = args.sym ? tiles.sym[width] : nullptr;
  const int nblocks = tiles_of(n, width, args.sym != 0, tiles);
  if (variant >= 1) {
    const CUtensorMap maps[8] = {mAhi, mAlo, mBhi, mBlo, mA2hi, mA2lo, mB2hi, mB2lo};
    return launch_persistent(s, width, maps, args, nblocks, nullptr, 0);
  }
  if (wide) {
    const int sb = smem_bytes<256>();
    const cudaError_t attr = ensure_smem(8, gemm_tc_kernel<256>, sb);
    if (attr != cudaSuccess) return attr;
    gemm_tc_kernel<256><<<nblocks, 192, sb, s>>>(mAhi, mAlo, mBhi, mBlo, mA2hi, mA2lo, mB2hi, mB2lo, args);
    note_launch();
  } else {
    const int sb = smem_bytes<128>();
    const cudaError_t attr = ensure_smem(9, gemm_tc_kernel<128>, sb);
    if (attr != cudaSuccess) return attr;
    gemm_tc_kernel<128><<<nblocks, 192, sb, s>>>(mAhi, mAlo, mBhi, mBlo, mA2hi, mA2lo, mB2hi, mB2lo, args);
    note_launch();
  }
  return cudaGetLastError();
}

struct TcGroupCache {
  std::unordered_map<uint64_t, TcEntry*> tables;
};

TcGroupCache* tc_group_cache_new() { return new TcGroupCache(); }

void tc_group_cache_free(TcGroupCache* c) {
  if (!c) return;
  for (auto& kv : c->tables) cudaFree(kv.second);
  delete c;
}

namespace {
inline uint64_t fnv_mix(uint64_t h, uint64_t x) {
  for (int i = 0; i < 8; ++i) {
    h ^= (x >> (8 * i)) & 0xff;
    h *= 1099511628211ull;
  }
  return h;
}
template <typename T>
inline uint64_t bits_of(T v) {
  uint64_t x = 0;
  std::memcpy(&x, &v, sizeof(T) < 8 ? sizeof(T) : 8);
  return x;
}
}  // namespace

cudaError_t gemm_tc_group(cudaStream_t s, int n, const TcProblem* probs, int nprob, TcArgs shared,
                          const TcTiles& tiles, TcGroupCache* cache) {
  if (nprob < 1 || !cache || shared.fmt < 0 || shared.fmt > 2) return cudaErrorInvalidValue;
  if (n % 128 != 0 || n <= 0 || (shared.pairs != 1 && shared.pairs != 2)) return cudaErrorInvalidValue;
  if (nprob == 1) {
    TcProblem one = probs[0];
    TcArgs& a = one.epi;
    a.nseg = shared.nseg;
    a.pairs = shared.pairs;
    a.sym = shared.sym;
    a.fmt = shared.fmt;
    a.split_acc = shared.split_acc;
    a.chunk_kb = shared.chunk_kb;
    a.err = shared.err;
    return gemm_tc(s, n, one, tiles);
  }
  const int width = pick_width(n, nprob, shared, tiles);
  const int bn = tc_width(width);
  // table key: the problems' operands and epilogue arguments (a table is rebuilt only when
  // one of them changes)
  uint64_t key = 1469598103934665603ull;
  key = fnv_mix(key, (uint64_t)n * 1000003u + shared.nseg * 7 + shared.pairs * 31 + shared.sym * 131 +
                         shared.fmt * 521 + (uint64_t)bn * 7919);
  key = fnv_mix(key, (uint64_t)(shared.sym ? tiles.sym[width] : nullptr));
  key = fnv_mix(key, (uint64_t)shared.err + (uint64_t)shared.chunk_kb);
  for (int i = 0; i < nprob; ++i) {
    const TcProblem& q = probs[i];
    const TcArgs& e = q.epi;
    const uint64_t w[] = {(uint64_t)q.Ahi, (uint64_t)q.Alo, (uint64_t)q.Bhi, (uint64_t)q.Blo, (uint64_t)q.A2hi,
                          (uint64_t)q.A2lo, (uint64_t)q.B2hi, (uint64_t)q.B2lo, (uint64_t)e.E,
                          (uint64_t)e.E2, (uint64_t)e.E64, (uint64_t)e.dvec, (uint64_t)e.out.f, (uint64_t)e.out.d,
                          (uint64_t)e.out.hi, (uint64_t)e.out.lo, (uint64_t)e.out.scale, (uint64_t)e.out2.f,
                          (uint64_t)e.out2.hi, (uint64_t)e.out2.lo, (uint64_t)e.out2.scale, (uint64_t)e.sa,
                          (uint64_t)e.sb, bits_of(e.alpha), bits_of(e.beta), bits_of(e.beta2), bits_of(e.beta64),
                          bits_of(e.diag), bits_of(e.dvec_scale), bits_of(e.va), bits_of(e.vb),
                          (uint64_t)e.ndvec * 17 + (uint64_t)e.ldc * 65537};
    for (uint64_t x : w) key = fnv_mix(key, x);
  }
  TcArgs a = shared;
  a.n = n;
  a.K = n;
  a.tiles_n = n / bn;
  a.tile_list = a.sym ? tiles.sym[width] : nullptr;
  const int tiles_per = tiles_of(n, width, a.sym != 0, tiles);
  TcEntry* table = nullptr;
  auto it = cache->tables.find(key);
  if (it != cache->tables.end()) {
    table = it->second;
  } else {
    std::vector<TcEntry> host(nprob);
    for (int i = 0; i < nprob; ++i) {
      const TcProblem& q = probs[i];
      TcEntry& t = host[i];
      const void* Alo = q.Alo ? q.Alo : q.Ahi;
      const void* Blo = q.Blo ? q.Blo : q.Bhi;
      if (!make_map(&t.map[0], q.Ahi, n, BM, shared.fmt) || !make_map(&t.map[1], Alo, n, BM, shared.fmt) ||
          !make_map(&t.map[2], q.Bhi, n, bn, shared.fmt) || !make_map(&t.map[3], Blo, n, bn, shared.fmt))
        return cudaErrorInvalidValue;
      if (shared.pairs == 2) {
        const void* r[4];
        second_pair(q, r);
        if (!make_map(&t.map[4], r[0], n, BM, shared.fmt) || !make_map(&t.map[5], r[1], n, BM, shared.fmt) ||
            !make_map(&t.map[6], r[2], n, bn, shared.fmt) || !make_map(&t.map[7], r[3], n, bn, shared.fmt))
          return cudaErrorInvalidValue;
      } else {
        t.map[4] = t.map[0];
        t.map[5] = t.map[1];
        t.map[6] = t.map[2];
        t.map[7] = t.map[3];
      }
      // the problem's epilogue arguments, with the launch's shared fields (the epilogue reads
      // sym, the kernel's walk n, K, nseg, pairs, ...)
      t.args = q.epi;
      t.args.n = a.n;
      t.args.K = a.K;
      t.args.nseg = a.nseg;
      t.args.pairs = a.pairs;
      t.args.sym = a.sym;
      t.args.fmt = a.fmt;
      t.args.split_acc = a.split_acc;
      t.args.chunk_kb = a.chunk_kb;
      t.args.tiles_n = a.tiles_n;
      t.args.tile_list = a.tile_list;
      t.args.err = a.err;
    }
    cudaError_t e = cudaMalloc((void**)&table, sizeof(TcEntry) * nprob);
    if (e != cudaSuccess) return e;
    // pageable source: the call returns once the bytes are staged, ordered on the stream
    e = cudaMemcpyAsync(table, host.data(), sizeof(TcEntry) * nprob, cudaMemcpyHostToDevice, s);
    if (e != cudaSuccess) {
      cudaFree(table);
      return e;
    }
    cache->tables[key] = table;
  }
  const int ntiles = nprob * tiles_per;
  // the launch's own maps are unused (every problem's maps come from the table)
  CUtensorMap dummy[8];
  std::memset(dummy, 0, sizeof(dummy));
  return launch_persistent(s, width, dummy, a, ntiles, table, tiles_per);
}

// Tile list of symmetric two-SM products: the 256 x 256 tiles (tm, tn) with tn >= tm, in the
// grouped raster of the dense products.
std::vector<int> tc_sym_tiles_pair(int n) {
  std::vector<int> t;
  const int tiles = n / 256;
  for (int first = 0; first < tiles; first += kPairGroupM) {
    const int gm = std::min(tiles - first, kPairGroupM);
    for (int tn = 0; tn < tiles; ++tn)
      for (int tm = first; tm < first + gm; ++tm)
        if (tn >= tm) {
          t.push_back(tm);
          t.push_back(tn);
        }
  }
  return t;
}

// Tile lists of symmetric products: tiles (tm, tn) of BM x bn that reach the
// upper triangle (bn tn + bn > BM tm), row-major order.
std::vector<int> tc_sym_tiles(int n, int bn) {
  std::vector<int> t;
  const int tiles_m = n / BM, tiles_n = n / bn;
  for (int first = 0; first < tiles_m; first += kGroupM) {
    const int gm = std::min(tiles_m - first, kGroupM);
    for (int tn = 0; tn < tiles_n; ++tn)
      for (int tm = first; tm < first + gm; ++tm)
        if (bn * tn + bn > BM * tm) {
          t.push_back(tm);
          t.push_back(tn);
        }
  }
  return t;
}

}  // namespace xl
