// Kernels of the superiorized simultaneous feasibility-seeking loop
// (arXiv 2509.20012, Sec. 2.4.3: Fig. 2 in simultaneous form, Fig. 3, Eq. 2)
// for sm_103a.  Memory-bound sparse work: no tensor cores.
//
//   K1 k_forward     fused Dx / Lx over one shared CSR index stream, 16-byte
//                    streaming loads of col / D / L, x staged in shared
//                    memory by one bulk (TMA) copy, warp per row, rows
//                    assigned to warps in nnz-balanced contiguous ranges;
//                    fused epilogues: objective residual (Eq. 2), line-search
//                    coefficients, FP64 final outputs.
//   K2 k_constraints per-row half-space evaluation and relaxed projection
//                    coefficients (Fig. 2), FP64 norms and divides.
//   K3 k_backward    transposed product over the CSC copy, split into
//                    fixed-size column chunks, one warp per chunk range;
//                    every chunk sum is a fixed-order warp reduction (no
//                    float atomics, deterministic).
//   K3b k_colfinish  per spot: sum of its chunks in order, then the
//                    gradient, or the clip w <- max(0, x + u) (Fig. 2, last
//                    loop); closes the iteration (log entry, k).
//   K4 k_finish      one block, or 64 and then the last one: deterministic
//                    reduction of the partials and the closed-form
//                    non-ascent trial loop (Fig. 3) in one warp.
//   K5 setup         in fredopt_load.cu (row order, values, CSC copy, tiles);
//                    here the based 16-bit row offsets of the CSC.
#include "fredopt.h"
#include "fredopt_internal.cuh"
#include "fredopt_device.cuh"

#include <algorithm>

#include <cstdio>
#include <type_traits>

namespace fo {

// Launch shape and streaming depth (compile-time; the defaults were chosen
// by measurement on GB300).
#ifndef FO_FWD_UNROLL
#define FO_FWD_UNROLL 1
#endif
#ifndef FO_BWD_UNROLL
#define FO_BWD_UNROLL 2
#endif
#ifndef FO_PREFETCH_UNITS
#define FO_PREFETCH_UNITS 1
#endif
#ifndef FO_BWD_MIN_BLOCKS
#define FO_BWD_MIN_BLOCKS 4
#endif
#ifndef FO_FWD_XS
#define FO_FWD_XS 1
#endif
#ifndef FO_FWD_THREADS
#define FO_FWD_THREADS 1024
#endif
constexpr int kFwdThreads = FO_FWD_THREADS;
constexpr int kFwdUnroll = FO_FWD_UNROLL;
#ifndef FO_UNROLL16
#define FO_UNROLL16 2
#endif
#ifndef FO_BWD_UNROLL16
#define FO_BWD_UNROLL16 3
#endif
#ifndef FO_BWD_PP
#define FO_BWD_PP 0
#endif
constexpr int kFwdUnroll16 = FO_UNROLL16;
// Register units (blocks of 128 elements loaded together) of the transposed
// product per pass: FO_BWD_UNROLL16 for the 16-bit projection pass (D and L
// streams), FO_BWD_UNROLL16_G for the 16-bit gradient pass (L stream only),
// FO_BWD_UNROLL_G for the FP32 gradient pass.  The gradient passes carry
// fewer bytes per element, so more of their elements fit in the 64
// registers of a thread.  Clinical plan, per launch (mean of both passes):
// BF16 0.598 -> 0.535 ms, FP32 0.687 -> 0.672 ms against 2/2/2 units.
#ifndef FO_BWD_UNROLL16_G
#define FO_BWD_UNROLL16_G 4
#endif
#ifndef FO_BWD_UNROLL_G
#define FO_BWD_UNROLL_G 3
#endif
// 1: a pass that uses only the L components of the coefficient pairs gathers
// 4 bytes per element instead of the 8-byte pair (fewer registers)
#ifndef FO_BWD_GATHER_Y
#define FO_BWD_GATHER_Y 1
#endif
template <typename VT, bool UD>
__host__ __device__ constexpr int bwd_units() {
  return sizeof(VT) == 4 ? (UD ? FO_BWD_UNROLL : FO_BWD_UNROLL_G) : (UD ? FO_BWD_UNROLL16 : FO_BWD_UNROLL16_G);
}
constexpr bool kBwdPingPong = FO_BWD_PP != 0;
constexpr int kPrefetchUnits = FO_PREFETCH_UNITS;
constexpr int kBwdThreads = 256;
constexpr int kRowThreads = 256;
constexpr int kConThreads = 64;
constexpr int kFinishOne = 1024;  // partials per array up to which one CTA forms the scalar finish
constexpr int kColThreads = 256;
constexpr int kMbarSpins = FREDOPT_WAIT_POLLS;
// Lane mapping of a block's 128 elements (element of value q of lane l):
//   0 contiguous  4l + q            (16-byte index / FP32 loads per lane)
//   1 strided     32q + l           (one gather instruction reads the
//                                    coefficients of 32 consecutive elements)
//   2 pairs       64(q/2) + 2l + q%2 (4-byte 16-bit loads; 64-element spans)
// The transposed product gathers a coefficient per element; consecutive CSC
// elements of a column are mostly neighbouring voxels, so mappings 1 and 2
// touch fewer L1 sectors per gather instruction.  Mapping 2 measured fastest
// for both value widths (clinical plan, per launch: FP32 0.687 ms against
// 0.707 strided and 0.728 contiguous; BF16 0.598 against 0.644 contiguous
// and 0.676 strided).
#ifndef FO_BWD_LM
#define FO_BWD_LM 2
#endif
#ifndef FO_BWD_LM16
#define FO_BWD_LM16 2
#endif
template <typename VT>
constexpr int kBwdLaneMap = sizeof(VT) == 4 ? FO_BWD_LM : FO_BWD_LM16;
template <int LM>
__device__ __forceinline__ int lane_pos(int lane, int q) {
  return LM == 0 ? lane * 4 + q : LM == 1 ? q * 32 + lane : (q >> 1) * 64 + 2 * lane + (q & 1);
}

// ------------------------------------------------------------------ helpers

template <typename VT> struct VecOf;
template <> struct VecOf<float> { static constexpr int V = 4; };
// 16-bit values: 4 per lane too (8-byte value loads), so a block keeps the
// register footprint of the FP32 block and more blocks fit in a unit
template <> struct VecOf<__nv_bfloat16> { static constexpr int V = 4; };
template <> struct VecOf<__half> { static constexpr int V = 4; };

// 16-byte loads of the streamed arrays.  S = streaming (read once):
// FO_LOAD_KIND 0: ld.global.cs (evict-first in L1 and L2);
//              1: ld.global.L1::no_allocate;
//              2: ld.global.L1::no_allocate with an L2 evict-first policy;
//              3: ld.global.nc.L1::no_allocate.
// Otherwise (data reused across passes while it fits in L2): ld.global.nc.
#ifndef FO_LOAD_KIND
#define FO_LOAD_KIND 0
#endif
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ int4 ld_stream(const int4* p) {
  int4 v;
#if FO_LOAD_KIND == 0
  v = __ldcs(p);
#elif FO_LOAD_KIND == 1
  asm volatile("ld.global.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
#elif FO_LOAD_KIND == 2
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.s32 {%0,%1,%2,%3}, [%4], %5;"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(l2_evict_first_policy()));
#else
  asm volatile("ld.global.nc.L1::no_allocate.v4.s32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
#endif
  return v;
}
template <bool S>
__device__ __forceinline__ int4 ld16(const int4* p) {
  if (S) return ld_stream(p);
  return __ldg(p);
}
template <bool S>
__device__ __forceinline__ uint4 ld16(const uint4* p) {
  if (S) {
    const int4 v = ld_stream(reinterpret_cast<const int4*>(p));
    return make_uint4((unsigned)v.x, (unsigned)v.y, (unsigned)v.z, (unsigned)v.w);
  }
  return __ldg(p);
}

__device__ __forceinline__ void unpack(float, uint4 u, float* o) {
  o[0] = __uint_as_float(u.x);
  o[1] = __uint_as_float(u.y);
  o[2] = __uint_as_float(u.z);
  o[3] = __uint_as_float(u.w);
}
// 16-bit values: 4 per lane in the low 8 bytes (u.x, u.y)
__device__ __forceinline__ void unpack(__nv_bfloat16, uint4 u, float* o) {
  const uint32_t w[2] = {u.x, u.y};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    o[2 * i] = __uint_as_float(w[i] << 16);
    o[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}
__device__ __forceinline__ void unpack(__half, uint4 u, float* o) {
  const uint32_t w[2] = {u.x, u.y};
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    __half2 h = *reinterpret_cast<const __half2*>(&w[i]);
    float2 f = __half22float2(h);
    o[2 * i] = f.x;
    o[2 * i + 1] = f.y;
  }
}

// ---- mbarrier + bulk copy (TMA engine, non-tensor form) ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// bulk prefetch of [src, src + bytes) into L2 (TMA engine; no registers or
// shared memory; bytes a multiple of 16, src 16-byte aligned)
__device__ __forceinline__ void bulk_prefetch_l2(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
// bounded wait on phase `parity`; true when the phase completed
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int max_spins) {
  const uint32_t a = smem_u32(bar);
  for (int i = 0; i < max_spins; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// ------------------------------------------------------------------ streaming core

// One block of the index stream and the two value streams, 4 elements per
// lane: 16 bytes of 32-bit indices (8 bytes of 16-bit ones, in c0.x, c0.y)
// and 16 bytes of FP32 values (8 bytes of 16-bit ones, in the low half).
template <typename VT>
struct Blk {
  int4 c0;      // 4 indices
  uint4 a, b;   // values of the two streams
  int hb;       // block header of based 16-bit indices (see BlockBase)
};

// Based 16-bit indices: the stream is cut into aligned blocks of 128
// elements; block k holds uint16 offsets from hdr[k] >= 0, or, when its
// indices span 65536 or more, hdr[k] = -1 - j and its 128 int32 indices are
// ovf[128 j .. 128 j + 127].
struct BlockBase {
  const int32_t* hdr;
  const int32_t* ovf;
  int32_t n_ovf;
};

struct SegCheck {
  int64_t n_elems;
  int* err;
};

template <bool S>
__device__ __forceinline__ int4 ld_idx(const int32_t* p) {
  return ld16<S>(reinterpret_cast<const int4*>(p));
}
template <bool S>
__device__ __forceinline__ int4 ld_idx(const uint16_t* p) {  // 4 x 16-bit = 8 bytes
  uint2 v;
  if (S) v = __ldcs(reinterpret_cast<const uint2*>(p));
  else v = __ldg(reinterpret_cast<const uint2*>(p));
  return make_int4((int)v.x, (int)v.y, 0, 0);
}
__device__ __forceinline__ void unpack_idx(int32_t, int4 c, int* cs) {
  cs[0] = c.x; cs[1] = c.y; cs[2] = c.z; cs[3] = c.w;
}
__device__ __forceinline__ void unpack_idx(uint16_t, int4 c, int* cs) {  // little-endian halves
  cs[0] = (int)((uint32_t)c.x & 0xffffu); cs[1] = (int)((uint32_t)c.x >> 16);
  cs[2] = (int)((uint32_t)c.y & 0xffffu); cs[3] = (int)((uint32_t)c.y >> 16);
}

template <bool S>
__device__ __forceinline__ uint4 ld_vals(const float* p) {
  return ld16<S>(reinterpret_cast<const uint4*>(p));
}
template <bool S, typename H>
__device__ __forceinline__ uint4 ld_vals(const H* p) {  // 4 x 16-bit = 8 bytes
  uint2 v;
  if (S) v = __ldcs(reinterpret_cast<const uint2*>(p));
  else v = __ldg(reinterpret_cast<const uint2*>(p));
  return make_uint4(v.x, v.y, 0u, 0u);
}

template <typename VT, bool S, bool USE_A, typename IT>
__device__ __forceinline__ void load_blk(Blk<VT>& k, const IT* idx, const VT* Av, const VT* Bv,
                                         int64_t p) {
  k.c0 = ld_idx<S>(idx + p);
  if (USE_A) k.a = ld_vals<S>(Av + p);
  k.b = ld_vals<S>(Bv + p);
}

// Lane-strided block: elements p, p + 32, p + 64, p + 96 (p = block start +
// lane), packed into the same registers as load_blk's 4 consecutive ones.
template <bool S, typename T>
__device__ __forceinline__ T ld1(const T* p) {
  if (S) return __ldcs(p);
  return __ldg(p);
}
template <bool S, typename T>
__device__ __forceinline__ uint4 ld_strided(const T* p) {
  if constexpr (sizeof(T) == 4) {
    const unsigned* q = reinterpret_cast<const unsigned*>(p);
    return make_uint4(ld1<S>(q), ld1<S>(q + 32), ld1<S>(q + 64), ld1<S>(q + 96));
  } else {
    const unsigned short* q = reinterpret_cast<const unsigned short*>(p);
    const uint32_t e0 = ld1<S>(q), e1 = ld1<S>(q + 32), e2 = ld1<S>(q + 64), e3 = ld1<S>(q + 96);
    return make_uint4(e0 | (e1 << 16), e2 | (e3 << 16), 0u, 0u);
  }
}
template <typename VT, bool S, bool USE_A, typename IT>
__device__ __forceinline__ void load_blk_strided(Blk<VT>& k, const IT* idx, const VT* Av, const VT* Bv,
                                                 int64_t p) {
  const uint4 c = ld_strided<S>(idx + p);
  k.c0 = make_int4((int)c.x, (int)c.y, (int)c.z, (int)c.w);
  if (USE_A) k.a = ld_strided<S>(Av + p);
  k.b = ld_strided<S>(Bv + p);
}
// Pair block: elements p, p + 1, p + 64, p + 65 (p = block start + 2 lane).
template <bool S, typename T>
__device__ __forceinline__ uint4 ld_pairs(const T* p) {
  if constexpr (sizeof(T) == 4) {
    const uint2* q = reinterpret_cast<const uint2*>(p);
    const uint2 a = ld1<S>(q), b = ld1<S>(q + 32);
    return make_uint4(a.x, a.y, b.x, b.y);
  } else {
    const unsigned* q = reinterpret_cast<const unsigned*>(p);
    return make_uint4(ld1<S>(q), ld1<S>(q + 32), 0u, 0u);
  }
}
template <typename VT, bool S, bool USE_A, typename IT>
__device__ __forceinline__ void load_blk_pairs(Blk<VT>& k, const IT* idx, const VT* Av, const VT* Bv,
                                               int64_t p) {
  const uint4 c = ld_pairs<S>(idx + p);
  k.c0 = make_int4((int)c.x, (int)c.y, (int)c.z, (int)c.w);
  if (USE_A) k.a = ld_pairs<S>(Av + p);
  k.b = ld_pairs<S>(Bv + p);
}

// Streams the elements [ptr[r0], ptr[r1]) of one warp as consecutive blocks
// of 32*V elements (lane l holds elements l*V .. l*V+V-1 of a block; every
// load is 16 bytes; the next unit of U blocks is in flight while the
// current one is consumed) and splits the stream into the segments
// [ptr[r], ptr[r+1]).  For element i with index c: sA += A_i * g(c).x and
// sB += B_i * g(c).y (in double-float for Acc = DF, four elements of a lane at
// a time).  A finished segment is summed over the warp in a fixed butterfly;
// lane (r - base) keeps it; every 32 segments (and at the end)
// flush(base, count, mine_A, mine_B) runs with lane j < count owning segment
// base + j.  Deterministic: the split depends only on ptr, r0, r1.  The index
// stream is int32 or uint16 (IT), the latter plain or BASED on per-block
// headers (bb); the sums do not depend on the encoding.  LM: lane mapping
// of a block's elements (lane_pos; mapping 0 is the one described above).
// The arrays must be readable (zero padded) up to
// round_up(ptr[r1], 32*V) + U*32*V elements (a prefetch starts below ptr[r1]
// and covers U*32*V elements, within the same bound).
// ready() runs when the first unit's loads are on their way and before the
// first gather: it waits for what the gathers read, and false ends the call.
struct NoWait {
  __device__ bool operator()() const { return true; }
};
template <typename VT, typename Acc, bool S, bool USE_A, int U, bool BASED = false, int LM = 0,
          typename IT, class Gather, class Flush, class Ready, int PF = kPrefetchUnits, bool PP = false>
__device__ __forceinline__ void stream_segments(const IT* __restrict__ idx,
                                                const VT* __restrict__ Av, const VT* __restrict__ Bv,
                                                const int64_t* __restrict__ ptr, int64_t r0, int64_t r1,
                                                int lane, Gather gather, Flush flush, Ready ready,
                                                BlockBase bbase = BlockBase{nullptr, nullptr, 0},
                                                SegCheck chk = SegCheck{0, nullptr}) {
  constexpr int V = VecOf<VT>::V;
  constexpr int BLK = 32 * V;
  constexpr int UB = U * BLK;
  static_assert(!BASED || (BLK == 128 && sizeof(IT) == 2), "based indices: 16-bit, 128-element blocks");
  if (r0 >= r1) return;
#if FO_CHECKED
  if (chk.err) {
    const int64_t p0 = ptr[r0], p1 = ptr[r1];
    if (p0 < 0 || p1 < p0 || (p1 + BLK - 1) / BLK * BLK + UB > chk.n_elems) {
      if (lane == 0) atomicOr(chk.err, 2);
      return;
    }
  }
#endif
  // 32-bit offsets from the block-aligned start of the warp's range (a
  // warp's range is far below 2^31 elements)
  const int64_t start = ptr[r0] & ~(int64_t)(BLK - 1);
  const int32_t* __restrict__ hdr = BASED ? bbase.hdr + start / BLK : nullptr;
  idx += start;
  if (USE_A) Av += start;
  Bv += start;
  const int pb = (int)(ptr[r0] - start), pe = (int)(ptr[r1] - start);
  const int nrows = (int)(r1 - r0);
  int row = 0, base = 0;  // relative to r0
  int ends = (lane < nrows) ? (int)(ptr[r0 + 1 + lane] - start) : pe;
  int e_cur = __shfl_sync(kFull, ends, 0);
  Acc sA{}, sB{}, myA{}, myB{};
  bool done = false;

  // consume the U blocks of one unit starting at offset b
  auto consume = [&](const Blk<VT>* unit, int b) {
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (done) return;
      const int bb = b + u * BLK;
      int cs[V];
      float av[V], bv[V];
      unpack_idx(IT(), unit[u].c0, cs);
      if (BASED) {
        const int hb = unit[u].hb;
        if (hb >= 0) {
#pragma unroll
          for (int q = 0; q < V; ++q) cs[q] += hb;
        } else {  // wide block: its int32 indices from the overflow table
          int slot = -1 - hb;
#if FO_CHECKED
          if (slot >= bbase.n_ovf) {
            if (chk.err) atomicOr(chk.err, 2);
            slot = 0;
          }
#endif
          const int32_t* ov = bbase.ovf + (int64_t)slot * BLK;
          if (LM == 1) {
#pragma unroll
            for (int q = 0; q < V; ++q) cs[q] = __ldg(ov + q * 32 + lane);
          } else if (LM == 2) {
            const int2 w0 = __ldg(reinterpret_cast<const int2*>(ov) + lane);
            const int2 w1 = __ldg(reinterpret_cast<const int2*>(ov + 64) + lane);
            cs[0] = w0.x; cs[1] = w0.y; cs[2] = w1.x; cs[3] = w1.y;
          } else {
            const int4 w = __ldg(reinterpret_cast<const int4*>(ov) + lane);
            cs[0] = w.x; cs[1] = w.y; cs[2] = w.z; cs[3] = w.w;
          }
        }
      }
      if (USE_A) unpack(VT(), unit[u].a, av);
      unpack(VT(), unit[u].b, bv);
      float2 gv[V];
#pragma unroll
      for (int q = 0; q < V; ++q) gv[q] = gather(cs[q]);
      int lo = bb > pb ? bb : pb;
      while (true) {
        const int hi = e_cur < bb + BLK ? e_cur : bb + BLK;
        if constexpr (std::is_same<Acc, DF>::value) {
          // elements outside [lo, hi) enter as 0 * 0
          static_assert(V == 4, "df_dot4");
          float am[V], bm[V], xm[V], ym[V];
#pragma unroll
          for (int q = 0; q < V; ++q) {
            const int e = bb + lane_pos<LM>(lane, q);
            const bool in = e >= lo && e < hi;
            am[q] = in ? av[q] : 0.0f;
            bm[q] = in ? bv[q] : 0.0f;
            xm[q] = in ? gv[q].x : 0.0f;
            ym[q] = in ? gv[q].y : 0.0f;
          }
          sA = df_dot4(am, xm, sA);
          sB = df_dot4(bm, ym, sB);
        } else {
#pragma unroll
          for (int q = 0; q < V; ++q) {
            const int e = bb + lane_pos<LM>(lane, q);
            if (e >= lo && e < hi) {
              if (USE_A) sA = fmaf(av[q], gv[q].x, sA);
              sB = fmaf(bv[q], gv[q].y, sB);
            }
          }
        }
        if (e_cur > bb + BLK) break;  // the open segment continues in the next block
        if (USE_A) {
          warp_sum2(sA, sB, lane);
        } else {
          sB = warp_sum(sB);
        }
        if (lane == row - base) { myA = sA; myB = sB; }
        sA = Acc{}; sB = Acc{};
        ++row;
        if (row - base == 32 || row == nrows) {
          flush(r0 + base, row - base, myA, myB);
          myA = Acc{}; myB = Acc{};
          if (row == nrows) { done = true; return; }
          base = row;
          ends = (base + lane < nrows) ? (int)(ptr[r0 + base + 1 + lane] - start) : pe;
        }
        e_cur = __shfl_sync(kFull, ends, row - base);
        lo = hi;
        if (lo >= bb + BLK) break;
      }
    }
  };
  // lane 0 asks the TMA engine to bring the unit PF units ahead into L2, so
  // the demand loads of the warp mostly wait on L2 rather than DRAM
  auto prefetch_unit = [&](int q) {
    if (PF > 0 && lane == 0 && q < pe) {
      bulk_prefetch_l2(idx + q, (uint32_t)(UB * sizeof(IT)));
      if (USE_A) bulk_prefetch_l2(Av + q, (uint32_t)(UB * sizeof(VT)));
      bulk_prefetch_l2(Bv + q, (uint32_t)(UB * sizeof(VT)));
    }
  };
  auto load_unit = [&](Blk<VT>* unit, int b) {
    prefetch_unit(b + PF * UB);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (LM == 1) load_blk_strided<VT, S, USE_A, IT>(unit[u], idx, Av, Bv, b + u * BLK + lane);
      else if (LM == 2) load_blk_pairs<VT, S, USE_A, IT>(unit[u], idx, Av, Bv, b + u * BLK + 2 * lane);
      else load_blk<VT, S, USE_A, IT>(unit[u], idx, Av, Bv, b + u * BLK + lane * V);
      if (BASED) unit[u].hb = __ldg(hdr + (b + u * BLK) / BLK);
    }
  };

  int b = 0;
#pragma unroll
  for (int k = 1; k < PF; ++k) prefetch_unit(b + k * UB);
  if (PP) {
    // ping-pong between two register units: while one is consumed the loads
    // of the other are in flight (no register copies of pending loads)
    Blk<VT> ua[U], ub[U];
    load_unit(ua, b);
    if (!ready()) return;
    while (true) {
      if (b + UB < pe) load_unit(ub, b + UB);
      consume(ua, b);
      if (done) break;
      b += UB;
      if (b + UB < pe) load_unit(ua, b + UB);
      consume(ub, b);
      if (done) break;
      b += UB;
    }
  } else {
    // one register unit: its U blocks are loaded together, then consumed;
    // latency is hidden by the other warps of the SM
    Blk<VT> ua[U];
    if constexpr (std::is_same<Ready, NoWait>::value) {
      while (!done) {
        load_unit(ua, b);
        consume(ua, b);
        b += UB;
      }
    } else {
      load_unit(ua, b);
      if (!ready()) return;
      while (true) {
        consume(ua, b);
        if (done) break;
        b += UB;
        load_unit(ua, b);
      }
    }
  }
}

// ------------------------------------------------------------------ K1

// Objective of one row (Eq. 2 terms of the structures the voxel is in):
// f_i = sum w (q - T)^2 ; residual rD = sum_DOSE 2w(Dx - T), rL = sum_CDL 2wc(cLx - T).
__device__ __forceinline__ void row_objective(const Tables& t, uint32_t m, double Dx, double Lx,
                                              double& f, double& rD, double& rL) {
  f = 0.0; rD = 0.0; rL = 0.0;
  for (int i = 0; i < t.n_obj; ++i) {
    const ObjEntry& o = t.obj[i];
    if (!((m >> o.bit) & 1u)) continue;
    if (o.q == 0) {
      const double d = Dx - o.target;
      f += o.weight * d * d;
      rD += 2.0 * o.weight * d;
    } else {
      const double d = t.c * Lx - o.target;
      f += o.weight * d * d;
      rL += 2.0 * o.weight * t.c * d;
    }
  }
}

template <typename IT> __device__ __forceinline__ const IT* fwd_col(const FwdArgs& a);
template <> __device__ __forceinline__ const int32_t* fwd_col<int32_t>(const FwdArgs& a) { return a.col; }
template <> __device__ __forceinline__ const uint16_t* fwd_col<uint16_t>(const FwdArgs& a) { return a.col16; }

// Fused Dx, Lx over the warp's nonempty rows [warp_row[2w], warp_row[2w+1]).
// IT: width of the column indices (uint16_t only with x in shared memory).
template <typename VT, int EPI, bool XS, bool S, typename IT>
__global__ void __launch_bounds__(kFwdThreads, 1024 / kFwdThreads) k_forward(FwdArgs a, Tables t) {
  extern __shared__ __align__(128) unsigned char smem[];
  using Acc = typename std::conditional<EPI == EPI_FINAL, DF, float>::type;
  const float* x = XS ? reinterpret_cast<const float*>(smem) : a.x;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem + fwd_bar_offset(a.n_x_pad));
  if (XS) {
    if (threadIdx.x == 0) {
      mbar_init(bar, 1);
      fence_mbar_init();
    }
    __syncthreads();
  }
  // Every warp runs this once: the predecessor has finished, and x is staged in
  // shared memory (by thread 0's bulk copy) unless the bounded wait gives up.
  // In passes that stay in L2 (S = false) a warp has its first loads on their way
  // by then (1.4% of the tiny plan's iteration; 0.2% slower in the long passes).
  bool waited = false, staged = true;
  auto ready = [&]() -> bool {
    if (waited) return staged;
    waited = true;
    pdl_wait();
    pdl_release();
    if (XS) {
      if (threadIdx.x == 0) {
        const uint32_t bytes = (uint32_t)a.n_x_pad * (uint32_t)sizeof(float);
        mbar_expect_tx(bar, bytes);
        bulk_g2s(smem, a.x, bytes, bar);
      }
      __syncwarp();
      staged = __all_sync(kFull, mbar_wait(bar, 0, kMbarSpins));
      if (!staged) {
        if ((threadIdx.x & 31) == 0) atomicOr(a.st->err, 1);
        mbar_wait(bar, 0, kMbarSpins);  // let the copy in flight land before leaving
      }
    }
    return staged;
  };
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  // Tiles: a warp streams tile `warp` (static schedule) or claims tiles in
  // order from a counter (a.sched[0]) until none is left, so that faster SMs
  // stream more of them; a.sched[1] counts the warps that are done and the
  // last one resets both counters for the next launch.  A tile's sums do not
  // depend on which warp streams it.
  auto claim = [&]() -> int {
    unsigned j = 0;
    if (lane == 0) j = atomicAdd(&a.sched[0], 1u);
    return (int)__shfl_sync(kFull, j, 0);
  };
  int job = a.sched ? claim() : warp;
  const VT* __restrict__ Dv = reinterpret_cast<const VT*>(a.Dv);
  const VT* __restrict__ Lv = reinterpret_cast<const VT*>(a.Lv);
  double acc0 = 0.0, acc1 = 0.0;  // per-lane partials of the epilogue reductions
  auto gather = [&](int c) {
    c = checked_index(c, a.n_x, a.st);
    const float v = x[c];
    return make_float2(v, v);
  };
  auto flush = [&](int64_t base, int cnt, Acc myD, Acc myL) {
    if (lane >= cnt) return;
    const int64_t r = base + lane;
    const float sd = a.sD ? a.sD[r] : 1.0f, sl = a.sL ? a.sL[r] : 1.0f;  // powers of two
    if constexpr (EPI == EPI_FINAL) {
      const double Dx = (double)myD * (double)sd, Lx = (double)myL * (double)sl;
      a.y64[r] = make_double2(Dx, Lx);
      const int64_t v = a.voxel ? a.voxel[r] : r;
      if (a.dose_out) a.dose_out[v] = (float)Dx;
      if (a.letd_out) a.letd_out[v] = Dx > 0.0 ? (float)(Lx / Dx) : 0.0f;
    } else {
      const float Dx = myD * sd, Lx = myL * sl;
      a.y[r] = make_float2(Dx, Lx);
      // FP64 only for rows with an objective term: GB300 issues an FP64 warp
      // instruction in about 15 cycles per SM, however few lanes are active,
      // and most warps hold no such row
      if constexpr (EPI == EPI_OBJ) {
        const uint32_t m = a.mask[r];
        float2 res = make_float2(0.0f, 0.0f);
        if (m & t.obj_bits) {
          double f, rD, rL;
          row_objective(t, m, Dx, Lx, f, rD, rL);
          res = make_float2((float)(rD * (double)sd), (float)(rL * (double)sl));
          acc0 += f;
        }
        a.r_out[r] = res;
      } else if constexpr (EPI == EPI_BC) {
        const uint32_t m = a.mask[r];
        if (m & t.obj_bits) {
          // B' = sum w (q(x) - T) q(g) = 1/2 (rD Dg + rL Lg); C' = sum w q(g)^2
          const float2 rin = a.r_in[r];  // already multiplied by the row scales
          acc0 += 0.5 * ((double)rin.x * (double)myD + (double)rin.y * (double)myL);
          double PD = 0.0, PL = 0.0;
          for (int i = 0; i < t.n_obj; ++i) {
            if (!((m >> t.obj[i].bit) & 1u)) continue;
            if (t.obj[i].q == 0) PD += t.obj[i].weight;
            else PL += t.obj[i].weight;
          }
          acc1 += PD * (double)Dx * (double)Dx + PL * t.c * t.c * (double)Lx * (double)Lx;
        }
      }
    }
  };
  if (S) ready();
  while (job < a.n_warps && staged) {
    // EPI_FINAL over listed rows: a tile is one row
    const bool one = EPI == EPI_FINAL && a.rows != nullptr;
    const int64_t r0 = one ? a.rows[job] : a.warp_row[2 * job], r1 = one ? r0 + 1 : a.warp_row[2 * job + 1];
    acc0 = 0.0;
    acc1 = 0.0;
    const auto stream = [&](auto before) {
      stream_segments<VT, Acc, S, true, (sizeof(VT) == 4 ? kFwdUnroll : kFwdUnroll16)>(
          fwd_col<IT>(a), Dv, Lv, a.rp, r0, r1, lane, gather, flush, before, BlockBase{nullptr, nullptr, 0},
          SegCheck{a.n_elems, FO_CHECKED ? a.st->err : nullptr});
    };
    if constexpr (S) stream(NoWait());
    else stream(ready);
    if ((EPI == EPI_OBJ || EPI == EPI_BC) && a.sched) {  // partials per tile, summed later in tile order
      const double s0 = warp_sum_nz(acc0), s1 = EPI == EPI_BC ? warp_sum_nz(acc1) : 0.0;
      if (lane == 0) {
        a.part[job] = s0;
        if (EPI == EPI_BC) a.part[a.part_stride + job] = s1;
      }
    }
    if (!a.sched) break;
    job = claim();
  }
  ready();  // a warp without rows waits too: no CTA leaves with the copy in flight
  if ((EPI == EPI_OBJ || EPI == EPI_BC) && !a.sched) {  // one tile per warp: a partial per CTA, in warp order
    const int wid = threadIdx.x >> 5;
    const double s0 = warp_sum_nz(acc0), s1 = EPI == EPI_BC ? warp_sum_nz(acc1) : 0.0;
    __syncthreads();  // x is not read any more
    double* red = reinterpret_cast<double*>(smem);
    static_assert(2 * 32 * sizeof(double) <= kFwdRedBytes && kFwdThreads <= 1024, "two sums per warp");
    if (lane == 0) {
      red[wid] = s0;
      red[32 + wid] = s1;
    }
    __syncthreads();
    if (wid < 2) {
      const double v = warp_sum_nz(lane < kFwdThreads / 32 ? red[32 * wid + lane] : 0.0);
      if (lane == 0 && (wid == 0 || EPI == EPI_BC)) a.part[wid * a.part_stride + blockIdx.x] = v;
    }
  }
  if (a.sched && lane == 0) {
    __threadfence();
    const unsigned total = (gridDim.x * blockDim.x) >> 5;
    if (atomicAdd(&a.sched[1], 1u) == total - 1) {
      a.sched[0] = 0u;
      a.sched[1] = 0u;
    }
  }
}



// ------------------------------------------------------------------ K3

// Chunk sums of the transposed product: chunk c = nonzeros [chunk_ptr[c],
// chunk_ptr[c+1]) of one column; sum_i D_ij coef_i.x + L_ij coef_i.y.
// NB: row indices as based 16-bit offsets (BwdArgs.row16/hdr/ovf).
template <typename VT, bool S, bool UD, bool NB>
__global__ void __launch_bounds__(kBwdThreads, FO_BWD_MIN_BLOCKS) k_backward(BwdArgs a) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const VT* __restrict__ Dv = reinterpret_cast<const VT*>(a.Dv);
  const VT* __restrict__ Lv = reinterpret_cast<const VT*>(a.Lv);
  const float2* cf = a.coef;  // the predecessor's output
  auto gather = [&](int r) {
    r = checked_index(r, a.n_rows, a.st);
    // plain loads: what a chained predecessor wrote is not read-only
    if (!UD && FO_BWD_GATHER_Y) return make_float2(0.0f, cf[r].y);
    return cf[r];
  };
  float* out = a.chunk_sum;
  auto flush = [&](int64_t base, int cnt, float mA, float mB) {
    if (lane < cnt) out[base + lane] = UD ? mA + mB : mB;
  };
  // tiles of column chunks, static (tile = warp) or claimed from a counter as
  // in the forward product; a chunk's sum does not depend on its warp
  auto claim = [&]() -> int {
    unsigned j = 0;
    if (lane == 0) j = atomicAdd(&a.sched[0], 1u);
    return (int)__shfl_sync(kFull, j, 0);
  };
  int job = a.sched ? claim() : warp;
  // (the first unit's loads ahead of the wait, as in the forward product, cost
  // registers that this kernel does not have)
  pdl_wait();
  pdl_release();
  while (job < a.n_warps) {
    if (NB)
      stream_segments<VT, float, S, UD, bwd_units<VT, UD>(), true, kBwdLaneMap<VT>,
                      uint16_t, decltype(gather), decltype(flush), NoWait, kPrefetchUnits, kBwdPingPong>(
          a.row16, Dv, Lv, a.chunk_ptr, a.warp_chunk[job], a.warp_chunk[job + 1], lane, gather, flush, NoWait(),
          BlockBase{a.hdr, a.ovf, a.n_ovf}, SegCheck{a.n_elems, FO_CHECKED ? a.st->err : nullptr});
    else
      stream_segments<VT, float, S, UD, bwd_units<VT, UD>(), false, kBwdLaneMap<VT>,
                      int32_t, decltype(gather), decltype(flush), NoWait, kPrefetchUnits, kBwdPingPong>(
          a.row, Dv, Lv, a.chunk_ptr, a.warp_chunk[job], a.warp_chunk[job + 1], lane, gather, flush, NoWait(),
          BlockBase{nullptr, nullptr, 0}, SegCheck{a.n_elems, FO_CHECKED ? a.st->err : nullptr});
    if (!a.sched) break;
    job = claim();
  }
  if (a.sched && lane == 0) {
    __threadfence();
    const unsigned total = (gridDim.x * blockDim.x) >> 5;
    if (atomicAdd(&a.sched[1], 1u) == total - 1) {
      a.sched[0] = 0u;
      a.sched[1] = 0u;
    }
  }
}

// ------------------------------------------------------------------ K3b

// The end of an iteration (block-wide): its log entry (violated rows and
// largest violation from the constraint partials, the solve state written by
// the scalar finish) and k <- k + 1.
__device__ __forceinline__ void close_iteration(const ColArgs& a, double* red) {
  const double nviol = block_count_array(a.k2part + a.k2_blocks, a.k2_blocks, red);
  const double mxv = block_max_array(a.k2part + 2 * a.k2_blocks, a.k2_blocks, red);
  if (threadIdx.x == 0) {
    DevState* st = a.st;
    if (st->log_cap > 0) {
      LogEntry e;
      e.k = st->k;
      e.s = st->s;
      e.accepted = st->accepted;
      e.n_violated = (int)nviol;
      e.beta = st->beta_acc;
      e.f_start = st->f_start;
      e.f_end = st->f_cur;
      e.gnorm = st->gnorm;
      e.max_violation = mxv;
      a.log[st->k % st->log_cap] = e;
    }
    st->k += 1;
  }
}

template <int MODE>
__global__ void __launch_bounds__(kColThreads) k_colfinish(ColArgs a) {
  __shared__ double red[kColThreads];
  __shared__ double sh_scale;
  __shared__ bool sh_last;
  // COL_PROJ with log_block: the launch's last block closes the iteration,
  // concurrently with the others (nothing else in the launch reads k), and
  // the other blocks split the columns
  const int nb = (int)gridDim.x - (MODE == COL_PROJ ? a.log_block : 0);
  pdl_wait();
  pdl_release();
  if (MODE == COL_PROJ && a.log_block && (int)blockIdx.x == nb) {
    close_iteration(a, red);
    return;
  }
  double scale = a.scale;  // COL_PROJ with has_scale: lam ps / W from the host
  if (MODE == COL_PROJ && !a.has_scale) {
    double W = a.W_all;
    if (a.norm == 1) W = block_sum_array(a.k2part, a.k2_blocks, red);
    if (threadIdx.x == 0) {
      const double ps = a.in_solve ? (a.st->eta == 1.0 ? 1.0 : pow(a.st->eta, (double)a.st->k)) : a.prio_scale;
      sh_scale = W > 0.0 ? a.lam * ps / W : 0.0;
    }
    __syncthreads();
    scale = sh_scale;
  }
  const double coef = (MODE == COL_PROJ && a.use_coef) ? a.st->coef : 0.0;
  const int per = (a.n + nb - 1) / nb;
  const int j0 = blockIdx.x * per, j1 = min(a.n, j0 + per);
  double acc = 0.0;
  for (int j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    float s = 0.0f;
    if (a.use_u) {
      // the chunk sums of the column in chunk order (loads unrolled ahead of
      // the sequential additions)
      const int c1 = a.col_chunk[j + 1];
#pragma unroll 8
      for (int c = a.col_chunk[j]; c < c1; ++c) s += __ldcg(&a.chunk_sum[c]);
    }
    if (MODE == COL_OUT) {
      a.out[j] = s;
    } else if (MODE == COL_GRAD) {
      a.out[j] = s;
      acc += (double)s * (double)s;
    } else {
      double xj = (double)a.w[j];
      if (a.use_coef) xj += coef * (double)a.g[j];
      const double wn = xj + scale * (double)s;
      a.w_out[j] = wn > 0.0 ? (float)wn : 0.0f;
    }
  }
  if (MODE == COL_GRAD) {
    acc = block_sum256(acc, red);
    if (threadIdx.x == 0) a.part[blockIdx.x] = acc;
  }
  if (MODE == COL_PROJ && a.in_solve && !a.log_block) {
    // the last block to finish closes the iteration: log entry, k <- k + 1
    __syncthreads();
    if (threadIdx.x == 0) {
      __threadfence();
      const unsigned prev = atomicAdd(&a.st->done, 1u);
      sh_last = (prev == gridDim.x - 1);
    }
    __syncthreads();
    if (sh_last) {
      __threadfence();
      close_iteration(a, red);
      if (threadIdx.x == 0) a.st->done = 0u;
    }
  }
}

// ------------------------------------------------------------------ K2

// (float)(g s) for a power of two s, as if scaled in FP64 and rounded once.  g itself
// is about 1 / |a_r|, which leaves the FP32 range for rows of very small or large
// values; where it and the product are normal FP32 numbers, scaling the rounded g is
// the same and takes no FP64 instruction (6e6 structure rows: 175 us, and 203 with
// the FP64 product everywhere).
__device__ __forceinline__ float scaled_coef(double g, float s) {
  if ((__double_as_longlong(g) << 1) == 0) return 0.0f;
  const float f = (float)g, r = f * s;
  auto normal = [](float v) { return ((__float_as_uint(v) >> 23) & 255u) - 1u < 254u; };
  return normal(f) && normal(r) ? r : (float)(g * (double)s);
}

// One listed row per thread and step.  Bound by FP64 instruction issue (an
// FP64 warp instruction holds an SM's pipe for about 15 cycles), so the rows are
// spread over CTAs of two warps and as many SMs as there are.
__global__ void __launch_bounds__(kConThreads) k_constraints(ConArgs a, Tables t) {
  constexpr int kWarps = kConThreads / 32;
  __shared__ ConEntry con[kMaxCon];
  __shared__ double wred[3][kWarps];
  __shared__ long long wcnt[kWarps];
  stage_constraints(t, con);
  __syncthreads();
  const int64_t step = (int64_t)gridDim.x * kConThreads;
  int64_t j = (int64_t)blockIdx.x * kConThreads + threadIdx.x;
  int64_t i = 0;
  uint32_t todo = 0u;
  double dd = 0.0, ll = 0.0, dl = 0.0;
  auto row = [&]() {  // what does not depend on the predecessor
    i = a.rows[j];
    todo = row_constraints(con, t.n_con, a.mask[i]);
    dd = a.dd[i];
    ll = a.ll[i];
    dl = a.dl[i];
  };
  if (j < a.n_list) row();
  pdl_wait();
  pdl_release();
  const double coef = a.use_coef ? a.st->coef : 0.0;
  double psum = 0.0, mx = 0.0, preach = 0.0;
  unsigned viol = 0u;
  while (j < a.n_list) {
    float2 out = make_float2(0.f, 0.f);
    if (todo) {
      const float2 w2 = a.yw[i];
      double xd = w2.x, xl = w2.y;
      if (a.use_coef) {
        const float2 g2 = a.yg[i];
        xd += coef * (double)g2.x;
        xl += coef * (double)g2.y;
      }
      double gD = 0.0, gL = 0.0;
      eval_constraints(con, todo, t.c, xd, xl, dd, ll, dl, gD, gL, psum, preach, viol, mx);
      out = a.sD ? make_float2(scaled_coef(gD, a.sD[i]), scaled_coef(gL, a.sL[i])) : make_float2((float)gD, (float)gL);
    }
    a.gam[i] = out;
    j += step;
    if (j < a.n_list) row();
  }
  // the block's two sums, its violated-row count and its largest violation
  // (>= 0): warp reductions (the FP64 butterflies skipped by warps without
  // violated or reachable rows), then the warp results in warp order
  psum = warp_sum_nz(psum);
  preach = warp_sum_nz(preach);
  const long long nv = (long long)__reduce_add_sync(kFull, viol);
  mx = warp_max_nonneg(mx);
  if ((threadIdx.x & 31) == 0) {
    const int wi = threadIdx.x >> 5;
    wred[0][wi] = psum;
    wred[1][wi] = preach;
    wred[2][wi] = mx;
    wcnt[wi] = nv;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    const int k = threadIdx.x;
    double r = wred[k == 0 ? 0 : k == 3 ? 1 : 2][0];
    long long c = wcnt[0];
#pragma unroll
    for (int w = 1; w < kWarps; ++w) {
      c += wcnt[w];
      if (k == 2) r = fmax(r, wred[2][w]);
      else if (k != 1) r += wred[k == 0 ? 0 : 1][w];
    }
    // partial slices: sum of priorities of violated rows, violated rows,
    // largest violation, sum of priorities of reachable rows
    a.part[k * gridDim.x + blockIdx.x] = k == 1 ? (double)c : r;
  }
}

// ------------------------------------------------------------------ K4

// The partial sums (one per forward tile: tens of thousands) are added in
// two fixed levels: every CTA sums one slice of each array, and the last CTA
// to finish adds the slice sums in order and runs the trial loop.  GB300's
// FP64 rate is low and an FP64 warp instruction costs the same with one
// active lane or 32, so each sum is laid out to need few of them: within a
// CTA, warps 2k and 2k + 1 add array k (lane l of warp 2k + h takes the
// elements 64 t + 32 h + l of the slice), each warp's lanes by a butterfly,
// the two warps' results in warp order; the last CTA adds the 64 slice sums
// of array k in warp k.  The solve state and the first trial steps are
// loaded at the start, so that the last CTA's chain of dependent loads is
// short.  With at most kFinishOne partials per array (one per forward CTA
// instead of one per claimed tile) a single CTA does it all.
__global__ void __launch_bounds__(256) k_finish(int step, const double* part_f, int nf,
                                                const double* part_bc, int nbc, const double* part_g,
                                                int ng, DevState* st, double* stage, const double* btab,
                                                long long n_btab) {
  __shared__ double wred[4][2];
  __shared__ double tot_sh[4];
  __shared__ bool sh_last;
  const int G = gridDim.x, b = blockIdx.x;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  // state read by the last CTA (written only by it, at its end, in this kernel)
  const long long s0 = st->s;
  const int max_trials = st->max_trials;
  const int grad_normalize = st->grad_normalize;
  const double f_empty = st->f_empty;
  double beta_pre = 0.0;  // step of trial `lane` (first round)
  if (wid == 0 && lane < max_trials) {
    const long long si = s0 + lane;
    if (si < n_btab) beta_pre = btab[si];
  }
  pdl_wait();
  pdl_release();
  {
    const int k = wid >> 1, h = wid & 1;
    const double* arr = k == 0 ? part_f : k == 1 ? part_bc : k == 2 ? part_bc + nbc : part_g;
    const int len = k == 0 ? nf : k == 3 ? ng : nbc;
    const int per = (len + G - 1) / G;
    const int i0 = min(len, b * per), i1 = min(len, i0 + per);
    double v = 0.0;
    for (int i = i0 + 32 * h + lane; i < i1; i += 64) v += arr[i];
    v = warp_sum_nz(v);
    if (lane == 0) wred[k][h] = v;
  }
  __syncthreads();
  if (G == 1) {
    if (threadIdx.x < 4) tot_sh[threadIdx.x] = wred[threadIdx.x][0] + wred[threadIdx.x][1];
  } else {
    if (threadIdx.x < 4) stage[threadIdx.x * G + b] = wred[threadIdx.x][0] + wred[threadIdx.x][1];
    if (threadIdx.x == 0) {
      __threadfence();
      sh_last = atomicAdd(&st->done_fin, 1u) == (unsigned)G - 1;
    }
    __syncthreads();
    if (!sh_last) return;
    __threadfence();
    // the slice sums, written by other CTAs of this launch: read past L1
    if (wid < 4) {
      double v = 0.0;
      for (int i = lane; i < G; i += 32) v += __ldcg(&stage[wid * G + i]);
      v = warp_sum_nz(v);
      if (lane == 0) tot_sh[wid] = v;
    }
  }
  __syncthreads();
  if (wid != 0) return;
  const double f = tot_sh[0] + (step == 0 ? f_empty : 0.0);
  const double Bp = tot_sh[1];
  const double Cp = tot_sh[2];
  const double gn2 = tot_sh[3];
  // The trial loop of Fig. 3 (beta = beta0 alpha^s, s advancing on every
  // trial, accept the first trial that does not ascend, at most max_trials):
  // the warp evaluates 32 consecutive trials at once, one per lane, and takes
  // the lowest accepting lane, so the decision and s are those of the trials
  // taken in turn.  The steps beta0 alpha^s come from the table filled at
  // fredopt_begin (s < n_btab), else from the same FP64 expression.
  const double gn = gn2 > 0.0 ? sqrt(gn2) : 0.0;
  const double ig = gn2 > 0.0 ? 1.0 / gn : 0.0;  // one FP64 division for B, C and the step
  double B = 0.0, C = 0.0;
  if (gn2 > 0.0) {
    if (grad_normalize) { B = -Bp * ig; C = Cp * ig * ig; }
    else { B = -Bp; C = Cp; }
  }
  int first = max_trials;  // index of the accepted trial, max_trials if none
  double beta_acc = 0.0;
  if (gn2 > 0.0) {
    for (int base = 0; base < max_trials; base += 32) {
      const int tr = base + lane;
      double beta = 0.0;
      bool ok = false;
      if (tr < max_trials) {
        const long long si = s0 + tr;
        beta = base == 0 && si < n_btab ? beta_pre
             : si < n_btab              ? btab[si]
                                        : st->beta0 * pow(st->alpha, (double)si);
        const double df = beta * (2.0 * B + beta * C);  // f(x + beta v) - f(x), Eq. 2 is quadratic
        ok = df <= 0.0;
      }
      const unsigned acc = __ballot_sync(kFull, ok);
      if (acc) {
        const int l = __ffs(acc) - 1;
        first = base + l;
        beta_acc = __shfl_sync(kFull, beta, l);
        break;
      }
    }
  }
  if (lane != 0) return;
  st->done_fin = 0u;
  if (step == 0) {
    st->f_start = f;
    st->accepted = 0;
    st->beta_acc = 0.0;
  }
  double fc = f;
  double coef = 0.0;
  long long s = s0;
  if (gn2 > 0.0) {
    st->gnorm = gn;
    if (first < max_trials) {
      const double beta = beta_acc;
      coef = grad_normalize ? -beta * ig : -beta;
      st->accepted += 1;
      st->accepted_total += 1;
      st->beta_acc = beta;
      fc = f + beta * (2.0 * B + beta * C);
      s = s0 + first + 1;
    } else {
      s = s0 + max_trials;
    }
  } else {
    st->gnorm = 0.0;
  }
  st->s = s;
  st->coef = coef;
  st->f_cur = fc;
}

// x <- x + coef g for the next perturbation step (reductions > 1)
__global__ void k_apply_step(int64_t n_hot, int n, float* w, const float* g, float2* yw,
                             const float2* yg, const DevState* st) {
  const double coef = st->coef;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) w[i] = (float)((double)w[i] + coef * (double)g[i]);
  if (i < n_hot) {
    const float2 a = yw[i], b = yg[i];
    yw[i] = make_float2((float)((double)a.x + coef * b.x), (float)((double)a.y + coef * b.y));
  }
}

__global__ void __launch_bounds__(kRowThreads) k_row_objective(Tables t, const float2* yw,
                                                              const uint32_t* mask, const float* sD,
                                                              const float* sL, int64_t n_hot,
                                                              float2* r_out, double* part) {
  __shared__ double red[kRowThreads];
  const int64_t per = (n_hot + gridDim.x - 1) / gridDim.x;
  const int64_t i0 = (int64_t)blockIdx.x * per, i1 = min(n_hot, i0 + per);
  double acc = 0.0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += blockDim.x) {
    const float2 y = yw[i];
    double f, rD, rL;
    row_objective(t, mask[i], y.x, y.y, f, rD, rL);
    const double sd = sD ? (double)sD[i] : 1.0, sl = sL ? (double)sL[i] : 1.0;
    r_out[i] = make_float2((float)(rD * sd), (float)(rL * sl));
    acc += f;
  }
  acc = block_sum256(acc, red);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// FP64 check at the final point over the listed rows (those with a structure
// bit): per block [max violation per kind (6), n violated, f]
__global__ void __launch_bounds__(kRowThreads) k_final_check(Tables t, const double2* y64,
                                                            const uint32_t* mask, const double* dd,
                                                            const double* ll, const double* dl,
                                                            const int64_t* rows, int64_t n_list, double* part) {
  __shared__ double red[kRowThreads];
  const int64_t per = (n_list + gridDim.x - 1) / gridDim.x;
  const int64_t j0 = (int64_t)blockIdx.x * per, j1 = min(n_list, j0 + per);
  double mk[6] = {0, 0, 0, 0, 0, 0};
  double nv = 0.0, fo = 0.0;
  for (int64_t j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    const int64_t i = rows[j];
    const uint32_t m = mask[i];
    const double2 y = y64[i];
    for (int q = 0; q < t.n_con; ++q) {
      const ConEntry& c = t.con[q];
      if (!((m >> c.bit) & 1u)) continue;
      const int fam = c.kind >> 1;
      double v, n2, b;
      if (fam == 0) { v = y.x; n2 = dd[i]; b = c.bound; }
      else if (fam == 1) { v = t.c * y.y; n2 = ll[i]; b = c.bound; }
      else {
        v = y.y - c.bound * y.x;
        n2 = ll[i] - 2.0 * c.bound * dl[i] + c.bound * c.bound * dd[i];
        b = 0.0;
      }
      if (!(n2 > 0.0)) continue;
      const double viol = (c.kind & 1) ? v - b : b - v;
      if (viol > 0.0) {
        nv += 1.0;
        const double vu = (fam == 2) ? (y.x > 0.0 ? viol / y.x : 0.0) : viol;
        mk[c.kind] = fmax(mk[c.kind], vu);
      }
    }
    double f, rD, rL;
    row_objective(t, m, y.x, y.y, f, rD, rL);
    fo += f;
  }
  for (int q = 0; q < 6; ++q) {
    const double v = block_max256(mk[q], red);
    if (threadIdx.x == 0) part[blockIdx.x * 8 + q] = v;
  }
  nv = block_sum256(nv, red);
  fo = block_sum256(fo, red);
  if (threadIdx.x == 0) {
    part[blockIdx.x * 8 + 6] = nv;
    part[blockIdx.x * 8 + 7] = fo;
  }
}

// Slice b of x (kSpotSlices slices): part[2 b] the sum of its squares, in the order
// that the host takes too (fredopt_api.cu, slice_squares); part[2 b + 1] twice the
// index of its first element that is not finite, or one more than that of its first
// negative one, whichever comes first; kNoSpot without either.
__global__ void __launch_bounds__(256) k_check_spots(const float* __restrict__ x, int32_t n, double* part) {
  __shared__ double red[9];
  __shared__ unsigned long long first;
  if (threadIdx.x == 0) first = kNoSpot;
  __syncthreads();
  const int per = (n + kSpotSlices - 1) / kSpotSlices;
  const int j0 = min((int64_t)n, (int64_t)blockIdx.x * per), j1 = min((int64_t)n, (int64_t)j0 + per);
  double sum = 0.0;
  for (int j = j0 + threadIdx.x; j < j1; j += 256) {
    const float v = x[j];
    if (!isfinite(v)) atomicMin(&first, 2ull * j);
    else if (v < 0.0f) atomicMin(&first, 2ull * j + 1ull);
    sum += (double)v * (double)v;
  }
  sum = block_sum256(sum, red);  // (its barriers order `first` too)
  if (threadIdx.x == 0) {
    part[2 * blockIdx.x] = sum;
    part[2 * blockIdx.x + 1] = (double)first;
  }
}

__global__ void __launch_bounds__(256) k_sum_slices(const double* __restrict__ part, int n, double* out) {
  __shared__ double red[9];
  const int per = (n + (int)gridDim.x - 1) / (int)gridDim.x;
  const int i0 = min(n, (int)blockIdx.x * per), i1 = min(n, i0 + per);
  const double v = block_sum_array(part + i0, i1 - i0, red);
  if (threadIdx.x == 0) out[blockIdx.x] = v;
}

// ------------------------------------------------------------------ K5 setup

template <typename VT>
__global__ void k_dequant_csc(const int64_t* cp, int32_t n_cols, const int32_t* row, const VT* DT,
                              const VT* LT, const float* sD, const float* sL, float* Dout, float* Lout) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; j < n_cols; j += nw) {
    for (int64_t p = cp[j] + lane; p < cp[j + 1]; p += 32) {
      const int r = row[p];
      Dout[p] = (sD ? sD[r] : 1.0f) * to_f(DT[p]);
      Lout[p] = (sL ? sL[r] : 1.0f) * to_f(LT[p]);
    }
  }
}

__global__ void k_scale_coef(int64_t n, const float* aD, const float* aL, const int64_t* voxel,
                             const float* sD, const float* sL, float2* coef) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t v = voxel ? voxel[i] : i;
  const float d = aD ? aD[v] : 0.0f, l = aL ? aL[v] : 0.0f;
  coef[i] = make_float2(sD ? d * sD[i] : d, sL ? l * sL[i] : l);
}


// reachable constraint rows (|a_r|^2 > 0) of the listed voxel rows: per block [count, unreachable, sum of priorities]
__global__ void __launch_bounds__(kRowThreads) k_count_rows(Tables t, const uint32_t* mask,
                                                           const double* dd, const double* ll,
                                                           const double* dl, const int64_t* rows,
                                                           int64_t n_list, double* part) {
  __shared__ double red[kRowThreads];
  const int64_t per = (n_list + gridDim.x - 1) / gridDim.x;
  const int64_t j0 = (int64_t)blockIdx.x * per, j1 = min(n_list, j0 + per);
  double nr = 0.0, nu = 0.0, W = 0.0;
  for (int64_t j = j0 + threadIdx.x; j < j1; j += blockDim.x) {
    const int64_t i = rows[j];
    const uint32_t m = mask[i];
    for (int q = 0; q < t.n_con; ++q) {
      const ConEntry& c = t.con[q];
      if (!((m >> c.bit) & 1u)) continue;
      const int fam = c.kind >> 1;
      const double n2 = fam == 0 ? dd[i]
                      : fam == 1 ? ll[i]
                                 : ll[i] - 2.0 * c.bound * dl[i] + c.bound * c.bound * dd[i];
      if (n2 > 0.0) { nr += 1.0; W += c.prio; }
      else nu += 1.0;
    }
  }
  nr = block_sum256(nr, red);
  nu = block_sum256(nu, red);
  W = block_sum256(W, red);
  if (threadIdx.x == 0) {
    part[3 * blockIdx.x] = nr;
    part[3 * blockIdx.x + 1] = nu;
    part[3 * blockIdx.x + 2] = W;
  }
}

__global__ void k_scatter_y(const float2* y, const int64_t* voxel, int64_t n, float* a, float* b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t v = voxel ? voxel[i] : i;
  const float2 t = y[i];
  if (a) a[v] = t.x;
  if (b) b[v] = t.y;
}

// ------------------------------------------------------------------ launch wrappers

// only the CTAs that hold scheduled warps (all of them for a full pass)
int forward_grid(const Geometry& g, int n_warps) {
  const int wpb = g.fwd_threads / 32;
  return std::max(1, std::min(g.fwd_blocks, (n_warps + wpb - 1) / wpb));
}

template <typename VT, int EPI, bool XS, bool S, typename IT = int32_t>
static void fwd_inst(const Geometry& g, const FwdArgs& a, const Tables& t, cudaStream_t s) {
  const size_t smem = XS ? fwd_bar_offset(a.n_x_pad) + kFwdBarBytes : kFwdRedBytes;
  launch_chain(a.pdl, k_forward<VT, EPI, XS, S, IT>, forward_grid(g, a.n_warps), g.fwd_threads, smem, s, a, t);
}

template <typename VT, int EPI>
static void fwd_dispatch_xs(const Geometry& g, bool xs, bool st, const FwdArgs& a, const Tables& t,
                            cudaStream_t s) {
  if (a.col16) {  // the load keeps 16-bit indices only when x fits shared memory
    if (EPI == EPI_FINAL || !st) fwd_inst<VT, EPI, true, false, uint16_t>(g, a, t, s);
    else fwd_inst<VT, EPI, true, true, uint16_t>(g, a, t, s);
    return;
  }
  if (EPI == EPI_FINAL) {
    if (xs) fwd_inst<VT, EPI, true, false>(g, a, t, s);
    else fwd_inst<VT, EPI, false, false>(g, a, t, s);
    return;
  }
  if (xs) {
    if (st) fwd_inst<VT, EPI, true, true>(g, a, t, s);
    else fwd_inst<VT, EPI, true, false>(g, a, t, s);
  } else {
    if (st) fwd_inst<VT, EPI, false, true>(g, a, t, s);
    else fwd_inst<VT, EPI, false, false>(g, a, t, s);
  }
}

template <typename VT>
static void fwd_dispatch_epi(const Geometry& g, int epi, bool xs, bool st, const FwdArgs& a,
                             const Tables& t, cudaStream_t s) {
  switch (epi) {
    case EPI_STORE: fwd_dispatch_xs<VT, EPI_STORE>(g, xs, st, a, t, s); break;
    case EPI_OBJ: fwd_dispatch_xs<VT, EPI_OBJ>(g, xs, st, a, t, s); break;
    case EPI_BC: fwd_dispatch_xs<VT, EPI_BC>(g, xs, st, a, t, s); break;
    default: fwd_dispatch_xs<VT, EPI_FINAL>(g, xs, st, a, t, s); break;
  }
}

bool forward_uses_smem(const Geometry& g, int n_x_pad) {
  return FO_FWD_XS && fwd_bar_offset(n_x_pad) + kFwdBarBytes <= g.smem_limit;
}

void launch_forward(const Geometry& g, int fmt, int epi, bool stream_hint, const FwdArgs& a,
                    const Tables& t, cudaStream_t s) {
  const bool xs = forward_uses_smem(g, a.n_x_pad);
  if (fmt == 1) fwd_dispatch_epi<__nv_bfloat16>(g, epi, xs, stream_hint, a, t, s);
  else if (fmt == 2) fwd_dispatch_epi<__half>(g, epi, xs, stream_hint, a, t, s);
  else fwd_dispatch_epi<float>(g, epi, xs, stream_hint, a, t, s);
}

template <typename VT, bool NB>
static void bwd_dispatch_nb(const Geometry& g, bool st, bool ud, const BwdArgs& a, cudaStream_t s) {
  if (st) {
    if (ud) launch_chain(a.pdl, k_backward<VT, true, true, NB>, g.bwd_blocks, g.bwd_threads, 0, s, a);
    else launch_chain(a.pdl, k_backward<VT, true, false, NB>, g.bwd_blocks, g.bwd_threads, 0, s, a);
  } else {
    if (ud) launch_chain(a.pdl, k_backward<VT, false, true, NB>, g.bwd_blocks, g.bwd_threads, 0, s, a);
    else launch_chain(a.pdl, k_backward<VT, false, false, NB>, g.bwd_blocks, g.bwd_threads, 0, s, a);
  }
}
template <typename VT>
static void bwd_dispatch(const Geometry& g, bool st, bool ud, const BwdArgs& a, cudaStream_t s) {
  if (a.row16) bwd_dispatch_nb<VT, true>(g, st, ud, a, s);
  else bwd_dispatch_nb<VT, false>(g, st, ud, a, s);
}

void launch_backward(const Geometry& g, int fmt, bool stream_hint, bool use_D, const BwdArgs& a,
                     cudaStream_t s) {
  if (fmt == 1) bwd_dispatch<__nv_bfloat16>(g, stream_hint, use_D, a, s);
  else if (fmt == 2) bwd_dispatch<__half>(g, stream_hint, use_D, a, s);
  else bwd_dispatch<float>(g, stream_hint, use_D, a, s);
}

int col_grid(const Geometry& g, int n) { return std::max(1, std::min(g.col_blocks, (n + 127) / 128)); }

void launch_colfinish(const Geometry& g, int mode, const ColArgs& a, cudaStream_t s) {
  const int grid = col_grid(g, a.n);
  if (mode == COL_OUT) launch_chain(a.pdl, k_colfinish<COL_OUT>, grid, kColThreads, 0, s, a);
  else if (mode == COL_GRAD) launch_chain(a.pdl, k_colfinish<COL_GRAD>, grid, kColThreads, 0, s, a);
  else launch_chain(a.pdl, k_colfinish<COL_PROJ>, grid + a.log_block, kColThreads, 0, s, a);
}

int con_grid(const Geometry& g, int64_t n_list) {
  // as many threads at most as row_blocks CTAs of the other row kernels have
  const int64_t cap = (int64_t)g.row_blocks * (kRowThreads / kConThreads);
  return (int)std::max<int64_t>(1, std::min<int64_t>(cap, (n_list + kConThreads - 1) / kConThreads));
}

void launch_constraints(const Geometry& g, const Tables& t, const ConArgs& a, cudaStream_t s) {
  launch_chain(a.pdl, k_constraints, con_grid(g, a.n_list), kConThreads, 0, s, a, t);
}

__global__ void k_beta_table(double* out, long long n, double beta0, double alpha) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = beta0 * pow(alpha, (double)i);
}

void launch_beta_table(double* out, long long n, double beta0, double alpha, cudaStream_t s) {
  if (n > 0) k_beta_table<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(out, n, beta0, alpha);
}

void launch_finish(int step, const double* part_f, int nf, const double* part_bc, int nbc,
                   const double* part_g, int ng, DevState* st, double* stage, const double* btab,
                   long long n_btab, bool pdl, cudaStream_t s) {
  const bool one = std::max(std::max(nf, nbc), ng) <= kFinishOne;
  launch_chain(pdl, k_finish, one ? 1 : kFinishBlocks, 256, 0, s, step, part_f, nf, part_bc, nbc, part_g, ng, st, stage, btab, n_btab);
}

void launch_apply_step(int64_t n_hot, int n, float* w, const float* g, float2* yw, const float2* yg,
                       const DevState* st, cudaStream_t s) {
  const int64_t m = n_hot > n ? n_hot : n;
  if (m == 0) return;
  k_apply_step<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(n_hot, n, w, g, yw, yg, st);
}

void launch_row_objective(const Geometry& g, const Tables& t, const float2* yw, const uint32_t* mask,
                          const float* sD, const float* sL, int64_t n_hot, float2* r_out,
                          double* part, cudaStream_t s) {
  k_row_objective<<<g.row_blocks, kRowThreads, 0, s>>>(t, yw, mask, sD, sL, n_hot, r_out, part);
}

void launch_final_check(int grid, const Tables& t, const double2* y64, const uint32_t* mask,
                        const double* dd, const double* ll, const double* dl, const int64_t* rows, int64_t n_list,
                        double* part, cudaStream_t s) {
  k_final_check<<<grid, kRowThreads, 0, s>>>(t, y64, mask, dd, ll, dl, rows, n_list, part);
}

void launch_check_spots(const float* x, int32_t n, double* part, cudaStream_t s) {
  k_check_spots<<<kSpotSlices, 256, 0, s>>>(x, n, part);
}

void launch_sum_slices(const double* part, int n, double* out, cudaStream_t s) {
  k_sum_slices<<<kFinishBlocks, 256, 0, s>>>(part, n, out);
}

void launch_count_rows(int grid, const Tables& t, const uint32_t* mask, const double* dd,
                       const double* ll, const double* dl, const int64_t* rows, int64_t n_list, double* part,
                       cudaStream_t s) {
  k_count_rows<<<grid, kRowThreads, 0, s>>>(t, mask, dd, ll, dl, rows, n_list, part);
}

void launch_scatter_y(const float2* y, const int64_t* voxel, int64_t n, float* a, float* b,
                      cudaStream_t s) {
  if (n == 0) return;
  k_scatter_y<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(y, voxel, n, a, b);
}

static unsigned grid_for(int64_t work, int per_block, int cap) {
  int64_t b = (work + per_block - 1) / per_block;
  if (b < 1) b = 1;
  if (b > cap) b = cap;
  return (unsigned)b;
}

void launch_dequant_csc(int fmt, const int64_t* cp, int32_t n_cols, const int32_t* row, const void* DT,
                        const void* LT, const float* sD, const float* sL, float* Dout, float* Lout,
                        cudaStream_t s) {
  const unsigned gb = grid_for(n_cols, 8, 65535);
  if (fmt == 1)
    k_dequant_csc<__nv_bfloat16><<<gb, 256, 0, s>>>(cp, n_cols, row, (const __nv_bfloat16*)DT,
                                                     (const __nv_bfloat16*)LT, sD, sL, Dout, Lout);
  else if (fmt == 2)
    k_dequant_csc<__half><<<gb, 256, 0, s>>>(cp, n_cols, row, (const __half*)DT, (const __half*)LT, sD,
                                              sL, Dout, Lout);
  else
    k_dequant_csc<float><<<gb, 256, 0, s>>>(cp, n_cols, row, (const float*)DT, (const float*)LT, sD,
                                             sL, Dout, Lout);
}

void launch_scale_coef(int64_t n, const float* aD, const float* aL, const int64_t* voxel,
                       const float* sD, const float* sL, float2* coef, cudaStream_t s) {
  if (n == 0) return;
  k_scale_coef<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, aD, aL, voxel, sD, sL, coef);
}

// ------------------------------------------------------------------ init

template <typename VT, int EPI, typename IT>
static cudaError_t set_smem_attr_it(int bytes) {
  cudaError_t e = cudaFuncSetAttribute(k_forward<VT, EPI, true, false, IT>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  if (EPI != EPI_FINAL)
    e = cudaFuncSetAttribute(k_forward<VT, EPI, true, true, IT>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  return e;
}
template <typename VT, int EPI>
static cudaError_t set_smem_attr(int bytes) {
  cudaError_t e = set_smem_attr_it<VT, EPI, int32_t>(bytes);
  if (e != cudaSuccess) return e;
  return set_smem_attr_it<VT, EPI, uint16_t>(bytes);
}

template <typename VT>
static cudaError_t set_smem_all(int bytes) {
  cudaError_t e;
  if ((e = set_smem_attr<VT, EPI_STORE>(bytes)) != cudaSuccess) return e;
  if ((e = set_smem_attr<VT, EPI_OBJ>(bytes)) != cudaSuccess) return e;
  if ((e = set_smem_attr<VT, EPI_BC>(bytes)) != cudaSuccess) return e;
  return set_smem_attr<VT, EPI_FINAL>(bytes);
}

cudaError_t kernel_arch(int* fwd_binary, int* bwd_binary, int* ptx_version) {
  cudaFuncAttributes fa, ba;
  cudaError_t e = cudaFuncGetAttributes(&fa, k_forward<float, EPI_OBJ, true, true, uint16_t>);
  if (e != cudaSuccess) return e;
  e = cudaFuncGetAttributes(&ba, k_backward<float, true, true, true>);
  if (e != cudaSuccess) return e;
  if (fwd_binary) *fwd_binary = fa.binaryVersion;
  if (bwd_binary) *bwd_binary = ba.binaryVersion;
  if (ptx_version) *ptx_version = fa.ptxVersion;
  return cudaSuccess;
}

int init_kernels(Geometry* g, int device) {
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return -1;
  g->n_sms = prop.multiProcessorCount;
  g->smem_limit = prop.sharedMemPerBlockOptin;
  g->fwd_threads = kFwdThreads;
  // 1024 threads per SM: one CTA when x is staged in shared memory (120 KB
  // for 30000 spots); smaller CTAs only when it is read through L1 instead
  g->fwd_blocks = g->n_sms * (FO_FWD_XS ? 1 : 1024 / kFwdThreads);
  g->fwd_warps = g->fwd_blocks * (kFwdThreads / 32);
  int occ = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_backward<float, true, true, false>, kBwdThreads, 0);
  if (occ < 1) occ = 1;
  g->bwd_threads = kBwdThreads;
  g->bwd_blocks = g->n_sms * occ;
  g->bwd_warps = g->bwd_blocks * (kBwdThreads / 32);
  g->row_threads = kRowThreads;
  g->row_blocks = g->n_sms * 4;
  g->col_threads = kColThreads;
  g->col_blocks = g->n_sms * 2;
  const int bytes = (int)g->smem_limit;
  if (set_smem_all<float>(bytes) != cudaSuccess) return -2;
  if (set_smem_all<__nv_bfloat16>(bytes) != cudaSuccess) return -2;
  if (set_smem_all<__half>(bytes) != cudaSuccess) return -2;
  if (init_load_kernels(bytes) != cudaSuccess || init_volume_kernels(bytes) != cudaSuccess) return -2;
  return 0;
}

// Based 16-bit row indices of the CSC (see BlockBase): one warp per block of
// 128 elements.  Pass 1 writes the block's base and offsets when its rows
// span less than 65536, else marks it -1 and counts it; pass 2 gives every
// marked block an overflow slot and copies its 128 int32 rows there.
__global__ void __launch_bounds__(256) k_narrow_rows(const int32_t* __restrict__ row, int64_t n_blk,
                                                     uint16_t* __restrict__ row16, int32_t* __restrict__ hdr,
                                                     unsigned int* n_wide) {
  const int lane = threadIdx.x & 31;
  const int64_t wstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n_blk; k += wstride) {
    const int4 v = __ldg(reinterpret_cast<const int4*>(row + k * 128) + lane);
    int lo = min(min(v.x, v.y), min(v.z, v.w)), hi = max(max(v.x, v.y), max(v.z, v.w));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(kFull, lo, o));
      hi = max(hi, __shfl_xor_sync(kFull, hi, o));
    }
    if ((int64_t)hi - (int64_t)lo < 65536) {
      reinterpret_cast<uint2*>(row16 + k * 128)[lane] =
          make_uint2((uint32_t)(v.x - lo) | ((uint32_t)(v.y - lo) << 16),
                     (uint32_t)(v.z - lo) | ((uint32_t)(v.w - lo) << 16));
      if (lane == 0) hdr[k] = lo;
    } else {
      reinterpret_cast<uint2*>(row16 + k * 128)[lane] = make_uint2(0u, 0u);
      if (lane == 0) {
        hdr[k] = -1;
        atomicAdd(n_wide, 1u);
      }
    }
  }
}

__global__ void __launch_bounds__(256) k_narrow_rows_wide(const int32_t* __restrict__ row, int64_t n_blk,
                                                          int32_t* __restrict__ hdr, int32_t* __restrict__ ovf,
                                                          unsigned int* slot, unsigned int n_wide) {
  const int lane = threadIdx.x & 31;
  const int64_t wstride = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < n_blk; k += wstride) {
    if (hdr[k] != -1) continue;
    unsigned j = 0;
    if (lane == 0) j = atomicAdd(slot, 1u);
    j = __shfl_sync(kFull, j, 0);
    if (j >= n_wide) continue;  // cannot happen: pass 1 counted every marked block
    reinterpret_cast<int4*>(ovf + (int64_t)j * 128)[lane] = __ldg(reinterpret_cast<const int4*>(row + k * 128) + lane);
    __syncwarp();
    if (lane == 0) hdr[k] = -1 - (int32_t)j;
  }
}

void launch_narrow_rows(const int32_t* row, int64_t n_blk, uint16_t* row16, int32_t* hdr, unsigned int* n_wide,
                        cudaStream_t s) {
  if (n_blk == 0) return;
  const unsigned grid = (unsigned)std::min<int64_t>((n_blk + 7) / 8, 152 * 8);
  k_narrow_rows<<<grid, 256, 0, s>>>(row, n_blk, row16, hdr, n_wide);
}

void launch_narrow_rows_wide(const int32_t* row, int64_t n_blk, int32_t* hdr, int32_t* ovf, unsigned int* slot,
                             unsigned int n_wide, cudaStream_t s) {
  if (n_blk == 0 || n_wide == 0) return;
  const unsigned grid = (unsigned)std::min<int64_t>((n_blk + 7) / 8, 152 * 8);
  k_narrow_rows_wide<<<grid, 256, 0, s>>>(row, n_blk, hdr, ovf, slot, n_wide);
}

// Failure detection without a fault: one CTA polls an mbarrier phase with the
// same bounded wait the bulk copies use.  With `arrive` set, thread 0 arrives
// first and the phase completes; otherwise nothing arrives, every poll fails,
// and after `spins` polls the CTA records the give-up in the error word and
// returns.  No copy is ever issued on this barrier.
__global__ void k_wait_check(int arrive, int spins, DevState* st) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (arrive && threadIdx.x == 0) mbar_expect_tx(&bar, 0u);
  if (!mbar_wait(&bar, 0, spins) && threadIdx.x == 0) atomicOr(st->err, 1);
}

void launch_wait_check(int arrive, int spins, DevState* st, cudaStream_t s) {
  k_wait_check<<<1, 32, 0, s>>>(arrive, spins > 0 ? spins : kMbarSpins, st);
}

}  // namespace fo
