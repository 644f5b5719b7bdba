// Tensor-core operands of the split precisions: hi = rn(x s), lo = rn(x s - hi) with a power-of-two
// scale s, rounded to FP16 or BF16 (16-bit words) or TF32 (an FP32 word whose low 13 mantissa bits are
// zero).  fmt: 0 FP16, 1 BF16, 2 TF32.
//
// The scale comes from a bound of |x| that is known before the matrix is computed, so whatever kernel
// computes it writes its operands too.  |x| s <= 2^14 keeps FP16 a factor of four from overflow; an
// element 2^-17 of the bound still keeps 22 bits, and below that the pair is good to 2^-39 of the bound.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace xl {

// 2^(14 - ceil(log2 bound)); 1 for a bound that is zero or not finite
__host__ __device__ inline float operand_scale(float bound) {
  if (!(bound > 0.0f) || !(bound < 1e37f)) return 1.0f;
  int e;
  frexpf(bound, &e);   // bound <= 2^e
  e = e < -40 ? -40 : e > 70 ? 70 : e;
  return ldexpf(1.0f, 14 - e);
}
__host__ __device__ inline float operand_scale(double bound) {
  // rounded up, so that it stays a bound; what FP32 cannot hold has the scale of the range's end
  return operand_scale(bound > 1e36 && bound < 1e300 ? 1e36f : (float)bound * 1.000001f);
}

// matrices that only matter against the identity (S, W, the residuals and their polynomials; all below 4)
constexpr float kUnitScale = 8192.0f;

template <int FMT>
struct OpWord {
  using T = unsigned short;
  using V4 = ushort4;
};
template <>
struct OpWord<2> {
  using T = unsigned;
  using V4 = uint4;
};

// Round x to the operand format; v receives the rounded value.  TF32 rounding (to 10 explicit
// mantissa bits, nearest, ties away from zero) is the cvt.rna.tf32.f32 instruction.
template <int FMT>
__device__ __forceinline__ typename OpWord<FMT>::T op_round(float x, float& v) {
  if constexpr (FMT == 2) {
    unsigned r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    v = __uint_as_float(r);
    return r;
  } else if constexpr (FMT == 1) {
    const __nv_bfloat16 b = __float2bfloat16_rn(x);
    v = __bfloat162float(b);
    return __bfloat16_as_ushort(b);
  } else {
    const __half h = __float2half_rn(x);
    v = __half2float(h);
    return __half_as_ushort(h);
  }
}

// Operands of four neighbouring values x + xl (xl: the low words of double-float values) at element i
// (a multiple of 4).  lo may be null.
template <int FMT>
__device__ __forceinline__ void store_operand4(void* hi, void* lo, size_t i, float s, const float (&x)[4],
                                               const float (&xl)[4]) {
  using T = typename OpWord<FMT>::T;
  using V4 = typename OpWord<FMT>::V4;
  T h[4], l[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float hv, lv;
    h[k] = op_round<FMT>(x[k] * s, hv);
    l[k] = op_round<FMT>((x[k] * s - hv) + xl[k] * s, lv);
  }
  V4 a;
  a.x = h[0]; a.y = h[1]; a.z = h[2]; a.w = h[3];
  *reinterpret_cast<V4*>(reinterpret_cast<T*>(hi) + i) = a;
  if (lo) {
    a.x = l[0]; a.y = l[1]; a.z = l[2]; a.w = l[3];
    *reinterpret_cast<V4*>(reinterpret_cast<T*>(lo) + i) = a;
  }
}

}  // namespace xl
