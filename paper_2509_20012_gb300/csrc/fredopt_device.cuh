// Device helpers shared by the kernels: warp sums and double-float arithmetic.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "fredopt_internal.cuh"

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
// Sums of two such values use the accurate
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
template <>
__device__ __forceinline__ DF warp_sum(DF v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const DF w(__shfl_xor_sync(kFull, v.hi, o), __shfl_xor_sync(kFull, v.lo, o));
    v = df_add(v, w);
  }
  return v;
}
// c + sum of four products in double-float: the products exact (TwoProd with an
// FMA: a x = p + fma(a, x, -p)), the three sums of their high parts exact (TwoSum),
// the seven error terms added in FP32, and joined to c by a TwoSum of the high parts
// and two FP32 additions.  With u = 2^-24 and M the four products' magnitudes, the
// error terms are at most 3 u M in all and pass three additions each, 8 u^2 M; the
// two that join them err by u^2 (|c| + 3 M) and u^2 (2 |c| + 4 M); when c and the sum
// nearly cancel, the last FastTwoSum's operands may lie the other way round, for no
// more than u^2 (|c| + 3 M) where the addition before it saves u^2 (|c| + M).  A
// step's error is at most 2^-48 (17 M + 3 |c|).  A row of n nonzeros takes n / 128
// steps per lane (two more where it starts and ends inside a block), and the lanes'
// sums are joined by five accurate additions, so
// its sum is within (3 n / 128 + 40) 2^-48 of its sum of magnitudes (absolutely: terms
// that cancel leave a larger relative error).  Four accurate double-word
// additions instead (88 FP32 operations, not 43; 3 u^2 of the partial sum each) bound
// it no better and measure the same or worse: largest errors in units of 2^-48 of the
// sum of magnitudes, four additions / this, over rows of
//   384 to 3072 nonzeros    positive 1.4 / 1.5   mixed signs 0.2 / 0.2   2^-30..2^30 1.0 / 0.9
//   58112 nonzeros          positive 2.2 / 2.1   mixed signs 0.1 / 0.1   2^-30..2^30 0.5 / 0.3
// The final pass is bound by these operations: 7.3e8 nonzeros, FP32 2.70 -> 1.46 ms,
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

// ------------------------------------------------------------------ checked builds

// Checked builds (FO_CHECKED=1, a debug aid in place of a memory checker): the
// kernels that stream the matrices check every tile's, row's and column's element
// range against the allocated length, every gathered index against its table and
// every overflow slot, record a failure in bit 1 of the error word (reported as
// FREDOPT_ERR_PATTERN) and skip the access.  Results are otherwise
// bit-identical to the default build.
#ifndef FO_CHECKED
#define FO_CHECKED 0
#endif
// i, or 0 with the failure recorded when i lies outside [0, n)
template <typename I>
__device__ __forceinline__ I checked_index(I i, int64_t n, const DevState* st) {
#if FO_CHECKED
  if ((int64_t)i < 0 || (int64_t)i >= n) {
    atomicOr(st->err, 2);
    return 0;
  }
#endif
  return i;
}
// e, or s with the failure recorded unless 0 <= s <= e <= n
__device__ __forceinline__ int64_t checked_end(int64_t s, int64_t e, int64_t n, const DevState* st) {
#if FO_CHECKED
  if (s < 0 || e < s || e > n) {
    atomicOr(st->err, 2);
    return s;
  }
#endif
  return e;
}

// ------------------------------------------------------------------ block reductions

// Block reductions of one double per thread (blockDim = 256), in a fixed
// order: a warp butterfly, then thread 0 adds the 8 warp results in warp
// order.  GB300 runs FP64 at a small fraction of its FP32 rate, and every
// FP64 warp instruction costs the same however few of its lanes are active,
// so: a warp whose lanes all hold zero skips its butterfly (its sum is that
// zero), maxima are of non-negative doubles, whose bit patterns order as
// signed 64-bit integers (integer compares), and counts held in doubles are
// added as 64-bit integers (exact, so in any order).
__device__ __forceinline__ double warp_sum_nz(double v) {
  if (!__any_sync(kFull, v != 0.0)) return v;
  return warp_sum(v);
}
__device__ __forceinline__ long long warp_max_bits(long long b) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long c = __shfl_xor_sync(kFull, b, o);
    b = c > b ? c : b;
  }
  return b;
}
__device__ __forceinline__ double warp_max_nonneg(double v) {
  return __longlong_as_double(warp_max_bits(__double_as_longlong(v)));
}
__device__ __forceinline__ long long warp_isum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}
// red: at least 9 doubles of shared memory; every thread returns the result
__device__ __forceinline__ double block_sum256(double v, double* red) {
  v = warp_sum_nz(v);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = red[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) r += red[w];
    red[8] = r;
  }
  __syncthreads();
  // red[8] is rewritten only after the next call's first barrier, which
  // every thread reaches after this read
  return red[8];
}
// v >= 0
__device__ __forceinline__ double block_max256(double v, double* red) {
  long long* rb = reinterpret_cast<long long*>(red);
  const long long b = warp_max_bits(__double_as_longlong(v));
  if ((threadIdx.x & 31) == 0) rb[threadIdx.x >> 5] = b;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long r = rb[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) r = rb[w] > r ? rb[w] : r;
    rb[8] = r;
  }
  __syncthreads();
  return __longlong_as_double(rb[8]);
}
// integers held in doubles (|v| < 2^53), added exactly
__device__ __forceinline__ double block_count256(long long v, double* red) {
  long long* rb = reinterpret_cast<long long*>(red);
  v = warp_isum(v);
  if ((threadIdx.x & 31) == 0) rb[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long r = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) r += rb[w];
    rb[8] = r;
  }
  __syncthreads();
  return (double)rb[8];
}
// Sum of n doubles in a fixed order (strided per thread, then block_sum256).
__device__ __forceinline__ double block_sum_array(const double* p, int n, double* red) {
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) v += p[i];
  return block_sum256(v, red);
}
// p[i] >= 0
__device__ __forceinline__ double block_max_array(const double* p, int n, double* red) {
  long long v = 0;
  for (int i = threadIdx.x; i < n; i += 256) {
    const long long b = __double_as_longlong(p[i]);
    v = b > v ? b : v;
  }
  return block_max256(__longlong_as_double(v), red);
}
__device__ __forceinline__ double block_count_array(const double* p, int n, double* red) {
  long long v = 0;
  for (int i = threadIdx.x; i < n; i += 256) v += (long long)p[i];
  return block_count256(v, red);
}

// ---- half-space evaluation of a voxel row (Fig. 2)
// |a_r|^2 of constraint c for a row with moments dd, ll, dl
__device__ __forceinline__ double row_norm2(const ConEntry& c, double cdl, double dd, double ll, double dl) {
  const int fam = c.kind >> 1;  // 0 dose, 1 cDL, 2 LETd
  return fam == 0 ? dd : fam == 1 ? cdl * cdl * ll : ll - 2.0 * c.bound * dl + c.bound * c.bound * dd;
}
// the constraint table in shared memory (a barrier follows at the caller)
__device__ __forceinline__ void stage_constraints(const Tables& t, ConEntry* con) {
  for (int q = threadIdx.x; q < t.n_con; q += blockDim.x) con[q] = t.con[q];
}
// bit q: constraint q applies to a voxel with structure mask m
__device__ __forceinline__ uint32_t row_constraints(const ConEntry* con, int n_con, uint32_t m) {
  uint32_t todo = 0u;
  for (int q = 0; q < n_con; ++q) todo |= ((m >> con[q].bit) & 1u) << q;
  return todo;
}
// Each lane walks the constraints of its own row, so a warp makes as many
// FP64 steps (a division or two each) as one of its rows has constraints, not
// as many as the table.  xd = (D x)_i, xl = (L x)_i; the sums run in table order.
__device__ __forceinline__ void eval_constraints(const ConEntry* con, uint32_t todo, double cdl, double xd, double xl,
                                                 double dd, double ll, double dl, double& gD, double& gL,
                                                 double& psum, double& preach, unsigned& nv, double& mx) {
  while (todo) {
    const ConEntry c = con[__ffs(todo) - 1];
    todo &= todo - 1u;
    const double n2 = row_norm2(c, cdl, dd, ll, dl);
    if (!(n2 > 0.0)) continue;  // unreachable row
    preach += c.prio;
    const int fam = c.kind >> 1;
    const double v = fam == 0 ? xd : fam == 1 ? cdl * xl : xl - c.bound * xd;
    const double b = fam == 2 ? 0.0 : c.bound;
    const double viol = (c.kind & 1) ? v - b : b - v;
    if (viol > 0.0) {
      const double tt = c.prio * (b - v) / n2;
      if (fam == 0) gD += tt;
      else if (fam == 1) gL += cdl * tt;
      else { gD -= c.bound * tt; gL += tt; }
      psum += c.prio;
      nv += 1u;
      const double vu = (fam == 2) ? (xd > 0.0 ? viol / xd : 0.0) : viol;  // LETd in keV/um
      mx = vu > mx ? vu : mx;
    }
  }
}

// ---- programmatic dependent launch
// A kernel launched as a link of a chain may start while its predecessor on the
// stream still runs.  It may read what no kernel of the chain writes at once;
// pdl_wait() returns when the predecessor has finished and its writes are
// visible (every thread calls it before it exits, so a chain stays ordered).
// Then pdl_release() lets the successor start.  What the chain writes is read
// with plain loads after the wait, never with the read-only path.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Launch as a link of such a chain (pdl), or ordered after the whole predecessor.
template <typename... P, typename... A>
void launch_chain(bool pdl, void (*kernel)(P...), unsigned grid, unsigned block, size_t smem, cudaStream_t s,
                  A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kernel, P(args)...);
}

}  // namespace fo
