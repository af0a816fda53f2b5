// Device helpers shared by the kernels: warp sums and double-float arithmetic.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace fo {

constexpr unsigned kFull = 0xffffffffu;

__device__ __forceinline__ float to_f(float v) { return v; }
__device__ __forceinline__ float to_f(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ __forceinline__ float to_f(__half v) { return __half2float(v); }

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// ---- double-float (double-word) accumulation ----
// A value hi + lo held in two FP32 numbers (|lo| <= ulp(hi) / 2): about 48
// significant bits at FP32 speed.  GB300's FP64 rate is a small fraction of
// its FP32 rate, so the final FP64-class pass accumulates in this form.
// Products are exact (TwoProd with an FMA); additions use the accurate
// double-word sum of Joldes, Muller and Popescu (ACM TOMS 44(2), 2017,
// relative error <= 3 * 2^-48), built from Knuth's TwoSum and Dekker's
// FastTwoSum.  Every operation is an explicitly rounded intrinsic, so the
// compiler cannot fuse or reorder any step.
struct DF {
  float hi, lo;
  __device__ DF() : hi(0.0f), lo(0.0f) {}
  __device__ explicit DF(float v) : hi(v), lo(0.0f) {}
  __device__ DF(float h, float l) : hi(h), lo(l) {}
  __device__ explicit operator double() const { return (double)hi + (double)lo; }
};
__device__ __forceinline__ DF two_sum(float a, float b) {
  const float s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
  return DF(s, e);
}
__device__ __forceinline__ DF fast_two_sum(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return DF(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ DF df_add(DF x, DF y) {
  const DF s = two_sum(x.hi, y.hi);
  const DF t = two_sum(x.lo, y.lo);
  const DF v = fast_two_sum(s.hi, __fadd_rn(s.lo, t.hi));
  return fast_two_sum(v.hi, __fadd_rn(t.lo, v.lo));
}
// c + a * b
__device__ __forceinline__ DF acc_fma(float a, float b, DF c) {
  const float p = __fmul_rn(a, b);
  return df_add(c, DF(p, __fmaf_rn(a, b, -p)));  // a * b = p + (a * b - p) exactly
}
template <>
__device__ __forceinline__ DF warp_sum(DF v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const DF w(__shfl_xor_sync(kFull, v.hi, o), __shfl_xor_sync(kFull, v.lo, o));
    v = df_add(v, w);
  }
  return v;
}
// c + sum of four products in double-float: the products exact (TwoProd), the
// three sums of their high parts exact (TwoSum), the seven error terms added
// in FP32, and one renormalised addition to c.  Against four acc_fma steps
// this is 43 FP32 operations instead of 88, and one rounding of the pair
// instead of four: over rows of 128 to 3072 nonzeros (positive, mixed-sign
// and wide-ranged values) its largest error against 64-bit-exact sums is the
// same or smaller (5e-15 against 6e-15 of the sum of magnitudes).  The final
// pass is bound by these operations: 7.3e8 nonzeros, FP32 2.70 -> 1.46 ms,
// FP16 2.59 -> 1.63 ms (its streaming floor is 1.07 and 0.65 ms).
__device__ __forceinline__ DF df_dot4(const float* a, const float* x, DF c) {
  float p[4], e[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    p[q] = __fmul_rn(a[q], x[q]);
    e[q] = __fmaf_rn(a[q], x[q], -p[q]);
  }
  const DF u = two_sum(p[0], p[1]), v = two_sum(p[2], p[3]);
  const DF s = two_sum(u.hi, v.hi);
  const float t = __fadd_rn(__fadd_rn(__fadd_rn(u.lo, v.lo), s.lo),
                            __fadd_rn(__fadd_rn(e[0], e[1]), __fadd_rn(e[2], e[3])));
  const DF w = two_sum(c.hi, s.hi);
  return fast_two_sum(w.hi, __fadd_rn(w.lo, __fadd_rn(c.lo, t)));
}

__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(kFull, v, o); }
__device__ __forceinline__ DF shfl_xor(DF v, int o) {
  return DF(__shfl_xor_sync(kFull, v.hi, o), __shfl_xor_sync(kFull, v.lo, o));
}
__device__ __forceinline__ float acc_add(float a, float b) { return a + b; }
__device__ __forceinline__ DF acc_add(DF a, DF b) { return df_add(a, b); }
// Both sums of a segment over the warp, bit for bit those of two butterflies
// (warp_sum): in the first step the lower half-warp takes over a and the upper
// one b, so the other four steps serve both; 6 shuffles and 5 additions
// instead of 10 and 10.
template <typename Acc>
__device__ __forceinline__ void warp_sum2(Acc& a, Acc& b, int lane) {
  const bool up = (lane & 16) != 0;
  const Acc give = up ? a : b;
  Acc keep = up ? b : a;
  keep = acc_add(keep, shfl_xor(give, 16));
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) keep = acc_add(keep, shfl_xor(keep, o));
  const Acc other = shfl_xor(keep, 16);
  a = up ? other : keep;
  b = up ? keep : other;
}

}  // namespace fo
