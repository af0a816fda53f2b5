// Kernels of the plan load (K5).  Everything that is proportional to the voxels
// or the nonzeros runs here; the host sees totals only.
//
//   k_rows_count,  device order of the rows: streamed rows with nonzeros, streamed
//   k_rows_scan,   rows without, other rows with and without (each ascending by
//   k_rows_place   voxel); their row pointers, masks and the list of structure rows
//   k_load_rows    one pass over the input: validation, index narrowing, value
//                  storage (quantised if asked) in device order, row moments
//   k_csc_count    per strip of rows: entries per column, and where each group
//                  of columns starts in every row (columns ascend in a row)
//   k_csc_colsum,  column totals over the strips; first output position of every
//   k_csc_offsets  (strip, column)
//   k_csc_fill     one CTA per (strip, column group) sorts tiles of entries by
//                  column in shared memory and writes them as runs
//   k_csc_scatter  the same for rows with very few entries per group
//   k_csc_columns, column pointers; the chunks of the transposed product
//   k_chunk_fill
//   k_tiles        bounds of the tiles that warps stream, by bisection of the
//                  row or chunk pointers
#include "fredopt_device.cuh"
#include "fredopt_internal.cuh"

#include <algorithm>
#include <climits>
#include <cmath>

namespace fo {

namespace {

// ------------------------------------------------------------------ row order

constexpr int kRowItems = 8;  // rows per thread
constexpr int kRowBlk = 256 * kRowItems;
constexpr int kRowCounters = 7;  // rows of groups 0, 1, 2; nonzeros of groups 0, 2; structure rows of groups 0, 1

// Group of row i: 0 streamed with nonzeros, 1 streamed without, 2 other with, 3 other without.
__device__ __forceinline__ int row_group(const int64_t* rp, const uint32_t* mask, int64_t i, int roi) {
  return ((!roi || mask[i] != 0u) ? 0 : 2) + (rp[i + 1] > rp[i] ? 0 : 1);
}

__global__ void __launch_bounds__(256) k_rows_count(const int64_t* __restrict__ rp, const uint32_t* __restrict__ mask,
                                                    int64_t n, int64_t nnz, int roi, int64_t* __restrict__ blk,
                                                    RowTotals* tot) {
  __shared__ unsigned long long sum[kRowCounters];
  __shared__ unsigned int bits[32];
  const int tid = threadIdx.x;
  if (tid < kRowCounters) sum[tid] = 0ull;
  if (tid < 32) bits[tid] = 0u;
  __syncthreads();
  unsigned flags = 0u;
  if (blockIdx.x == 0 && tid == 0 && (rp[0] != 0 || rp[n] != nnz)) flags |= kRowsBadEnds;
  unsigned c[kRowCounters] = {0u, 0u, 0u, 0u, 0u, 0u, 0u};
  long long z0 = 0, z2 = 0, zc = 0;
  for (int k = 0; k < kRowItems; ++k) {
    const int64_t i = (int64_t)blockIdx.x * kRowBlk + k * 256 + tid;
    if (i >= n) break;
    const int64_t len = rp[i + 1] - rp[i];
    const uint32_t m = mask[i];
    const int g = row_group(rp, mask, i, roi);
    if (len < 0) flags |= kRowsNotMonotone;
    if (i > 0 && row_group(rp, mask, i - 1, roi) > g) flags |= kRowsPermuted;
    c[0] += g == 0;
    c[1] += g == 1;
    c[2] += g == 2;
    c[5] += g == 0 && m != 0u;
    c[6] += g == 1 && m != 0u;
    if (g == 0) z0 += len;
    if (g == 0 && m != 0u) zc += len;
    if (g == 2) z2 += len;
    if (g == 1)
      for (uint32_t b = m; b; b &= b - 1u) atomicAdd(&bits[__ffs(b) - 1], 1u);
  }
#pragma unroll
  for (int j = 0; j < kRowCounters; ++j) {
    if (j == 3 || j == 4) {
      const long long z = warp_sum(j == 3 ? z0 : z2);
      if ((tid & 31) == 0 && z) atomicAdd(&sum[j], (unsigned long long)z);
    } else {
      const unsigned v = __reduce_add_sync(kFull, c[j]);
      if ((tid & 31) == 0 && v) atomicAdd(&sum[j], (unsigned long long)v);
    }
  }
  zc = warp_sum(zc);
  if ((tid & 31) == 0 && zc) atomicAdd(&tot->con_nnz, (unsigned long long)zc);
  flags = __reduce_or_sync(kFull, flags);
  if ((tid & 31) == 0 && flags) atomicOr(&tot->flags, flags);
  __syncthreads();
  if (tid < kRowCounters) blk[(int64_t)tid * gridDim.x + blockIdx.x] = (int64_t)sum[tid];
  if (tid < 32 && bits[tid]) atomicAdd(&tot->empty_bits[tid], (unsigned long long)bits[tid]);
}

// Warp c turns counter c of the blocks into exclusive prefixes.
__global__ void __launch_bounds__(kRowCounters * 32) k_rows_scan(int64_t* blk, int64_t nb, RowTotals* tot) {
  const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
  int64_t* p = blk + (int64_t)c * nb;
  int64_t run = 0;
  for (int64_t b0 = 0; b0 < nb; b0 += 128) {
    int64_t v[4];  // four consecutive blocks per lane
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = b0 + 4 * lane + k < nb ? p[b0 + 4 * lane + k] : 0;
    const int64_t own = v[0] + v[1] + v[2] + v[3];
    int64_t x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += y;
    }
    int64_t before = run + x - own;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (b0 + 4 * lane + k < nb) p[b0 + 4 * lane + k] = before;
      before += v[k];
    }
    run += __shfl_sync(kFull, x, 31);
  }
  if (lane == 0) tot->c[c] = run;
}

// Exclusive prefix of v over a block of 256 threads (wsum: 8 values).
__device__ __forceinline__ unsigned long long block_prefix256(unsigned long long v, unsigned long long* wsum) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  unsigned long long before = 0;
  for (int w = 0; w < wid; ++w) before += wsum[w];
  return before + x - v;
}

__global__ void __launch_bounds__(256) k_rows_place(const int64_t* __restrict__ rp, const uint32_t* __restrict__ mask,
                                                    int64_t n, int roi, const int64_t* __restrict__ blk,
                                                    const RowTotals* __restrict__ tot, int64_t* __restrict__ rp_out,
                                                    int64_t* __restrict__ voxel, uint32_t* __restrict__ mask_out,
                                                    int64_t* __restrict__ con_rows, float* __restrict__ sD,
                                                    float* __restrict__ sL) {
  __shared__ unsigned long long w1[8], w2[8];
  const int64_t i0 = (int64_t)blockIdx.x * kRowBlk + (int64_t)threadIdx.x * kRowItems;
  const int64_t i1 = min(n, i0 + kRowItems);
  // the five row counts of a block fit 12 bits each, its nonzeros 32 bits each
  unsigned long long rows = 0ull, nz = 0ull;
  for (int64_t i = i0; i < i1; ++i) {
    const int g = row_group(rp, mask, i, roi);
    const bool m = mask[i] != 0u;
    if (g < 3) rows += 1ull << (12 * g);
    if (g < 2 && m) rows += 1ull << (36 + 12 * g);
    if (g == 0) nz += (unsigned long long)(rp[i + 1] - rp[i]);
    if (g == 2) nz += (unsigned long long)(rp[i + 1] - rp[i]) << 32;
  }
  rows = block_prefix256(rows, w1);
  nz = block_prefix256(nz, w2);
  auto base = [&](int c) { return blk[(int64_t)c * gridDim.x + blockIdx.x]; };
  int64_t k0 = base(0) + (int64_t)(rows & 0xfffu), k1 = base(1) + (int64_t)((rows >> 12) & 0xfffu);
  int64_t k2 = base(2) + (int64_t)((rows >> 24) & 0xfffu);
  int64_t z0 = base(3) + (int64_t)(nz & 0xffffffffu), z2 = base(4) + (int64_t)(nz >> 32);
  int64_t q0 = base(5) + (int64_t)((rows >> 36) & 0xfffu), q1 = base(6) + (int64_t)((rows >> 48) & 0xfffu);
  const int64_t n0 = tot->c[0], n1 = tot->c[1], n2 = tot->c[2], nz0 = tot->c[3], nz2 = tot->c[4];
  for (int64_t i = i0; i < i1; ++i) {
    const int g = row_group(rp, mask, i, roi);
    const uint32_t m = mask[i];
    int64_t r, p;
    if (g == 0) {
      r = k0++;
      p = z0;
      z0 += rp[i + 1] - rp[i];
      if (m) con_rows[q0++] = r;
    } else if (g == 1) {
      r = n0 + k1++;
      p = nz0;
      if (m) con_rows[tot->c[5] + q1++] = r;
    } else if (g == 2) {
      r = n0 + n1 + k2++;
      p = nz0 + z2;
      z2 += rp[i + 1] - rp[i];
    } else {
      r = n0 + n1 + n2 + (i - k0 - k1 - k2);
      p = nz0 + nz2;
    }
    rp_out[r] = p;
    if (voxel) voxel[r] = i;
    if (g < 2) mask_out[r] = m;
    if (sD) sD[r] = sL[r] = 1.0f;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) rp_out[n] = nz0 + nz2;
}

// ------------------------------------------------------------------ input pass

// Power-of-two scale so that scale * q is exact in binary32:
// BF16: max|q| in (1/2, 1]; FP16: max|q| in (2^13, 2^14] (all normal values
// down to 2^-28 of the row maximum keep 11 significant bits).
__device__ __forceinline__ float pow2_scale(float amax, bool half) {
  if (!(amax > 0.0f)) return 1.0f;
  int ex;
  frexpf(amax, &ex);  // amax in [2^(ex-1), 2^ex)
  return ldexpf(1.0f, half ? ex - 14 : ex);
}

__device__ __forceinline__ void store_as(float v, float* q) { *q = v; }
__device__ __forceinline__ void store_as(float v, __nv_bfloat16* q) { *q = __float2bfloat16_rn(v); }
__device__ __forceinline__ void store_as(float v, __half* q) { *q = __float2half_rn(v); }

// One pass over the nonempty rows of the input (warp per row, device order):
//   - col strictly increasing in [0, n_cols), values finite (*err: 1, 2);
//   - indices to col_out, 16- or 32-bit;
//   - values to Dv, Lv in their storage type, 16-bit ones after a power-of-two
//     row scale (COPY = false: the input arrays are the storage already);
//   - for streamed rows the moments |D_i|^2, |L_i|^2, <D_i, L_i> of the stored
//     values in double-float (exact products; error bound at df_dot4), scales
//     applied at the end, exactly.
// Bound by its bytes: 12 read and 10 written per FP32 nonzero, 2.50 ms for
// 7.3e8 (6.4 TB/s).  Separate passes (validation 1.49 ms, row gather 5.87,
// moments 2.06, index narrowing 0.66) took 10.1 ms.
constexpr int kInK = 4;  // chunks of 32 entries in flight per warp

template <typename VT, typename IT, bool COPY>
__global__ void __launch_bounds__(256) k_load_rows(LoadRowsArgs a) {
  constexpr bool Q = sizeof(VT) == 2;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  IT* __restrict__ col_out = reinterpret_cast<IT*>(a.col_out);
  VT* __restrict__ Dv = reinterpret_cast<VT*>(a.Dv);
  VT* __restrict__ Lv = reinterpret_cast<VT*>(a.Lv);
  const int64_t jobs = a.n_hot_ne + a.n_cold_ne;
  for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < jobs; k += nw) {
    const int64_t r = k < a.n_hot_ne ? k : a.n_hot + (k - a.n_hot_ne);
    const int64_t i = a.voxel ? a.voxel[r] : r;
    const int64_t s = a.rp_in[i], d = a.rp_out[r];
    const int len = (int)(a.rp_in[i + 1] - s);
    const int32_t* __restrict__ ci = a.col + s;
    const float* __restrict__ Di = a.D + s;
    const float* __restrict__ Li = a.L + s;
    float scD = 1.0f, scL = 1.0f;
    if (Q) {
      float mD = 0.0f, mL = 0.0f;
      for (int j0 = lane; j0 < len; j0 += 32 * kInK) {
        float x[kInK], y[kInK];
#pragma unroll
        for (int q = 0; q < kInK; ++q) {
          const int j = j0 + 32 * q;
          x[q] = j < len ? Di[j] : 0.0f;
          y[q] = j < len ? Li[j] : 0.0f;
        }
#pragma unroll
        for (int q = 0; q < kInK; ++q) {
          mD = fmaxf(mD, fabsf(x[q]));
          mL = fmaxf(mL, fabsf(y[q]));
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        mD = fmaxf(mD, __shfl_xor_sync(kFull, mD, o));
        mL = fmaxf(mL, __shfl_xor_sync(kFull, mL, o));
      }
      scD = pow2_scale(mD, std::is_same<VT, __half>::value);
      scL = pow2_scale(mL, std::is_same<VT, __half>::value);
    }
    const bool hot = r < a.n_hot;
    int bad = 0, last = -1;
    DF mdd, mll, mdl;
    for (int j0 = 0; j0 < len; j0 += 32 * kInK) {
      int c[kInK];
      float x[kInK], y[kInK];
#pragma unroll
      for (int q = 0; q < kInK; ++q) {
        const int j = j0 + 32 * q + lane;
        const bool in = j < len;
        c[q] = in ? ci[j] : INT_MAX;
        x[q] = in ? Di[j] : 0.0f;
        y[q] = in ? Li[j] : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < kInK; ++q) {
        const int j = j0 + 32 * q + lane;
        int before = __shfl_up_sync(kFull, c[q], 1);
        if (lane == 0) before = last;
        last = __shfl_sync(kFull, c[q], 31);
        if (j < len) {
          if (c[q] < 0 || c[q] >= a.n_cols || before >= c[q]) bad |= 1;
          if (!isfinite(x[q]) || !isfinite(y[q])) bad |= 2;
          col_out[d + j] = (IT)c[q];
          if (Q) {
            VT qd, ql;
            store_as(x[q] / scD, &qd);
            store_as(y[q] / scL, &ql);
            Dv[d + j] = qd;
            Lv[d + j] = ql;
            x[q] = to_f(qd);
            y[q] = to_f(ql);
          } else if (COPY) {
            store_as(x[q], Dv + d + j);
            store_as(y[q], Lv + d + j);
          }
        }
      }
      if (hot) {
        mdd = df_dot4(x, x, mdd);
        mll = df_dot4(y, y, mll);
        mdl = df_dot4(x, y, mdl);
      }
    }
    bad = __reduce_or_sync(kFull, bad);
    if (bad && lane == 0) atomicOr(a.err, bad);
    if (Q && lane == 0) {
      a.sD[r] = scD;
      a.sL[r] = scL;
    }
    if (hot) {
      warp_sum2(mdd, mll, lane);
      mdl = warp_sum(mdl);
      if (lane == 0) {
        const double sd = (double)scD, sl = (double)scL;
        a.dd[r] = (double)mdd * (sd * sd);
        a.ll[r] = (double)mll * (sl * sl);
        a.dl[r] = (double)mdl * (sd * sl);
      }
    }
  }
}

// ------------------------------------------------------------------ counts

template <typename IT>
__device__ __forceinline__ int lower_bound_col(const IT* __restrict__ col, int len, int key) {
  int lo = 0, hi = len;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if ((int)col[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

constexpr int kCountThreads = 1024;
constexpr int kCountK = 8;

// Strip b = rows [strip_row[b], strip_row[b + 1]); cnt[b][c] = its entries in
// column c (SMEM: a shared-memory histogram, written once; else cnt starts at
// zero).  With `split`, split[r * (n_grp + 1) + q] = entries of row r before
// column q << gshift, for q = 0 .. n_grp (the last one is the row's length).
template <bool SMEM, typename IT>
__global__ void __launch_bounds__(kCountThreads) k_csc_count(const int64_t* __restrict__ rp,
                                                             const IT* __restrict__ col,
                                                             const int64_t* __restrict__ strip_row, int32_t n_cols,
                                                             int gshift, int n_grp,
                                                             int32_t* __restrict__ cnt, int32_t* __restrict__ split) {
  extern __shared__ int32_t sh_cnt[];
  const int lane = threadIdx.x & 31;
  int32_t* out = cnt + (int64_t)blockIdx.x * n_cols;
  int32_t* hist = SMEM ? sh_cnt : out;
  if (SMEM) {
    for (int j = threadIdx.x; j < n_cols; j += kCountThreads) sh_cnt[j] = 0;
    __syncthreads();
  }
  const int64_t r1 = strip_row[blockIdx.x + 1];
  for (int64_t r = strip_row[blockIdx.x] + (threadIdx.x >> 5); r < r1; r += kCountThreads / 32) {
    const int64_t s = rp[r];
    const int len = (int)(rp[r + 1] - s);
    const IT* __restrict__ cc = col + s;
    for (int i0 = lane; i0 < len; i0 += 32 * kCountK) {
      int c[kCountK];  // the loads of kCountK chunks in flight
#pragma unroll
      for (int k = 0; k < kCountK; ++k) c[k] = i0 + 32 * k < len ? (int)cc[i0 + 32 * k] : -1;
#pragma unroll
      for (int k = 0; k < kCountK; ++k)
        if (c[k] >= 0) atomicAdd(&hist[c[k]], 1);
    }
    // one group boundary per lane, found in the row just read
    if (split)
      for (int q = lane; q <= n_grp; q += 32)
        split[r * (n_grp + 1) + q] = q < n_grp ? lower_bound_col(cc, len, q << gshift) : len;
  }
  if (SMEM) {
    __syncthreads();
    for (int j = threadIdx.x; j < n_cols; j += kCountThreads) out[j] = sh_cnt[j];
  }
}

__global__ void k_csc_colsum(const int32_t* __restrict__ cnt, int n_strip, int32_t n_cols, int64_t* tot) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_cols) return;
  int64_t s = 0;
#pragma unroll 8
  for (int b = 0; b < n_strip; ++b) s += cnt[(int64_t)b * n_cols + j];
  tot[j] = s;
}

// cnt[b][j] <- first output position of strip b's entries of column j
__global__ void k_csc_offsets(int32_t* __restrict__ cnt, int n_strip, int32_t n_cols, const int64_t* __restrict__ cp) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_cols) return;
  int64_t run = cp[j];
  int b = 0;
  for (; b + 8 <= n_strip; b += 8) {  // eight loads in flight ahead of the running sum
    int32_t t[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) t[k] = cnt[(int64_t)(b + k) * n_cols + j];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      cnt[(int64_t)(b + k) * n_cols + j] = (int32_t)run;  // positions < 2^31 (checked on the host)
      run += t[k];
    }
  }
  for (; b < n_strip; ++b) {
    const int32_t t = cnt[(int64_t)b * n_cols + j];
    cnt[(int64_t)b * n_cols + j] = (int32_t)run;
    run += t;
  }
}

// ------------------------------------------------------------------ fill

// One CTA moves the entries of strip b in columns [g << gshift, (g + 1) << gshift)
// to their places, up to 32 rows (and T entries) at a time:
//   1  every entry sets its row's bit in its column's 32-bit mask (atomic OR:
//      any order);
//   2  a prefix over the columns' bit counts gives each column's first slot of
//      the tile;
//   3  an entry goes to slot first[c] + (rows of the tile before its own that
//      hold column c), its bits below its own in the mask: row order, so the
//      transpose is stable, with no order among the threads;
//   4  slot i of column c goes to output delta[c] + i.
// A column's entries are neighbours in the tile and in the output, so 32 stores
// of a warp touch a few runs instead of 32 places in each of the three arrays:
// scattered stores (their number, not their bytes) are what binds a transpose
// that stores entry by entry.  The CTAs that run at one time write a few
// groups' column frontiers, which stay in L2 until their lines are full.  With
// `split` a row's piece of the group is looked up, else found by bisection.
// 7.3e8 FP32 nonzeros: 8.3 ms, where 16-row steps with one 16-byte record
// store per entry and a pass to split the records took 17.7 ms.  Bound by the
// barriers and load latencies of its short tiles (a row has about 140 entries in
// an occupied group) and by frontier lines that leave L2 half full.  Four CTAs of
// 384 threads per SM: 8.3 ms; three of 512 8.5, four of 256 8.7, two of 768 14.8;
// groups of 512 columns 11.4, of 2048 10.1.
constexpr int kFillThreads = 384;
constexpr int kFillCtas = 4;       // per SM
constexpr int kFillGroupShift = 10;
constexpr int kFillWarps = kFillThreads / 32;
constexpr int kFillK = 5;  // chunks of 32 entries of a row in flight per warp

// the two values of an entry as one shared-memory word
template <typename VT> struct ValPair;
template <> struct ValPair<float> {
  using T = float2;
  static __device__ __forceinline__ T make(float d, float l) { return make_float2(d, l); }
  static __device__ __forceinline__ float d(T p) { return p.x; }
  static __device__ __forceinline__ float l(T p) { return p.y; }
};
template <> struct ValPair<uint16_t> {
  using T = uint32_t;
  static __device__ __forceinline__ T make(uint16_t d, uint16_t l) { return (uint32_t)d | ((uint32_t)l << 16); }
  static __device__ __forceinline__ uint16_t d(T p) { return (uint16_t)(p & 0xffffu); }
  static __device__ __forceinline__ uint16_t l(T p) { return (uint16_t)(p >> 16); }
};

template <typename VT>
struct FillSmem {  // byte offsets for T slots and G columns
  size_t val, rc, mask, first, delta, cur, off, src, scan, bytes;
  __host__ __device__ FillSmem(int T, int G) {
    size_t o = 0;
    auto take = [&](size_t b) { const size_t at = o; o = (o + b + 15) & ~(size_t)15; return at; };
    val = take(2 * sizeof(VT) * (size_t)T);
    rc = take(4 * (size_t)T);  // column << 5 | row of the tile
    mask = take(4 * (size_t)G);
    first = take(2 * (size_t)G);
    delta = take(4 * (size_t)G);
    cur = take(4 * (size_t)G);
    off = take(4 * (size_t)(kFillThreads + 1));
    src = take(8 * (size_t)kFillThreads);
    scan = take(4 * (size_t)kFillWarps);
    bytes = o;
  }
};

// Exclusive prefix of v over the block's threads; *total = the sum.  The
// caller has a barrier between two calls.
__device__ __forceinline__ int block_excl_scan(int v, int* wsum, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) wsum[wid] = x;
  __syncthreads();
  int before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kFillWarps; ++w) {
    const int t = wsum[w];
    if (w < wid) before += t;
    all += t;
  }
  *total = all;
  return before + x - v;
}

template <typename VT, typename IT>
__global__ void __launch_bounds__(kFillThreads) k_csc_fill(
    const int64_t* __restrict__ rp, const IT* __restrict__ col, const VT* __restrict__ Dv,
    const VT* __restrict__ Lv, const int64_t* __restrict__ strip_row, int n_strip, int32_t n_cols, int gshift, int n_grp,
    int T, const int32_t* __restrict__ split, const int32_t* __restrict__ cursor, int32_t* __restrict__ row_out,
    VT* __restrict__ DT, VT* __restrict__ LT) {
  extern __shared__ __align__(16) unsigned char fill_sh[];
  const int G = 1 << gshift;
  const FillSmem<VT> m(T, G);
  using VP = ValPair<VT>;
  typename VP::T* sVal = reinterpret_cast<typename VP::T*>(fill_sh + m.val);
  uint32_t* sRC = reinterpret_cast<uint32_t*>(fill_sh + m.rc);
  uint32_t* mask = reinterpret_cast<uint32_t*>(fill_sh + m.mask);
  uint16_t* first = reinterpret_cast<uint16_t*>(fill_sh + m.first);
  int32_t* delta = reinterpret_cast<int32_t*>(fill_sh + m.delta);
  int32_t* cur = reinterpret_cast<int32_t*>(fill_sh + m.cur);
  int32_t* off = reinterpret_cast<int32_t*>(fill_sh + m.off);
  int64_t* src = reinterpret_cast<int64_t*>(fill_sh + m.src);
  int* scan = reinterpret_cast<int*>(fill_sh + m.scan);
  const int b = blockIdx.x % n_strip, g = blockIdx.x / n_strip;
  const int c_base = g << gshift;
  const int gc = min(G, n_cols - c_base);  // columns of this group
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int j = tid; j < G; j += kFillThreads) {
    cur[j] = j < gc ? cursor[(int64_t)b * n_cols + c_base + j] : 0;
    mask[j] = 0u;
  }
  const int64_t r1 = strip_row[b + 1];
  for (int64_t r = strip_row[b]; r < r1; r += kFillThreads) {
    // ---- the pieces of the next rows: starts and running lengths
    const int n = (int)min((int64_t)kFillThreads, r1 - r);
    int len = 0;
    int64_t at = 0;
    if (tid < n) {
      const int64_t s = rp[r + tid];
      int a, e;
      if (split) {
        a = split[(r + tid) * (n_grp + 1) + g];
        e = split[(r + tid) * (n_grp + 1) + g + 1];
      } else {
        const int l = (int)(rp[r + tid + 1] - s);
        a = lower_bound_col(col + s, l, c_base);
        e = a + lower_bound_col(col + s + a, l - a, c_base + gc);
      }
      len = e - a;
      at = s + a;
    }
    int all;
    const int before = block_excl_scan(len, scan, &all);
    if (tid < n) {
      off[tid] = before;
      src[tid] = at;
    }
    if (tid == n - 1) off[n] = all;
    __syncthreads();
    if (all == 0) continue;  // off and scan are rewritten after the next barrier pair
    for (int j0 = 0; j0 < n;) {
      // the rows of this tile: at most 32, and what fits T (a piece is at most G <= T)
      const int base0 = off[j0];
      const int j1 = j0 + __popc(__ballot_sync(kFull, j0 + lane < n && off[min(j0 + lane + 1, n)] - base0 <= T));
      const int total = off[j1] - base0;
      if (total == 0) {
        j0 = j1;
        continue;
      }
      // ---- 1: the rows that hold each column
      for (int j = j0 + wid; j < j1; j += kFillWarps) {
        const int l = off[j + 1] - off[j];
        const IT* cc = col + src[j];
        const uint32_t bit = 1u << (j - j0);
        for (int i0 = 0; i0 < l; i0 += 32 * kFillK) {
          int c[kFillK];
#pragma unroll
          for (int q = 0; q < kFillK; ++q) c[q] = i0 + 32 * q + lane < l ? (int)cc[i0 + 32 * q + lane] - c_base : -1;
#pragma unroll
          for (int q = 0; q < kFillK; ++q)
            if (c[q] >= 0) atomicOr(&mask[c[q]], bit);
        }
      }
      __syncthreads();
      // ---- 2: first slot of every column (two neighbouring columns at a time)
      {
        const int pairs = G / 2;
        const int ppt = (pairs + kFillThreads - 1) / kFillThreads;
        const int k0 = tid * ppt, k1 = min(pairs, k0 + ppt);
        const uint2* mask2 = reinterpret_cast<const uint2*>(mask);
        int sum = 0;
        for (int k = k0; k < k1; ++k) {
          const uint2 w = mask2[k];
          sum += __popc(w.x) + __popc(w.y);
        }
        int t2;
        int slot = block_excl_scan(sum, scan, &t2);
        for (int k = k0; k < k1; ++k) {
          const uint2 w = mask2[k];
          const int n0 = __popc(w.x), n1 = __popc(w.y);
          const int2 p = reinterpret_cast<int2*>(cur)[k];
          reinterpret_cast<uint32_t*>(first)[k] = (uint32_t)slot | ((uint32_t)(slot + n0) << 16);
          reinterpret_cast<int2*>(delta)[k] = make_int2(p.x - slot, p.y - (slot + n0));
          reinterpret_cast<int2*>(cur)[k] = make_int2(p.x + n0, p.y + n1);
          slot += n0 + n1;
        }
      }
      __syncthreads();
      // ---- 3: entries to their slots
      for (int j = j0 + wid; j < j1; j += kFillWarps) {
        const int l = off[j + 1] - off[j];
        const int64_t p0 = src[j];
        const uint32_t below = (1u << (j - j0)) - 1u;
        for (int i0 = 0; i0 < l; i0 += 32 * kFillK) {
          int c[kFillK];
          VT d[kFillK], v[kFillK];
#pragma unroll
          for (int q = 0; q < kFillK; ++q) {
            const int i = i0 + 32 * q + lane;
            c[q] = -1;
            if (i < l) {
              c[q] = (int)col[p0 + i] - c_base;
              d[q] = Dv[p0 + i];
              v[q] = Lv[p0 + i];
            }
          }
#pragma unroll
          for (int q = 0; q < kFillK; ++q)
            if (c[q] >= 0) {
              const int pos = first[c[q]] + __popc(mask[c[q]] & below);
              sVal[pos] = VP::make(d[q], v[q]);
              sRC[pos] = ((uint32_t)c[q] << 5) | (uint32_t)(j - j0);
            }
        }
      }
      __syncthreads();
      // ---- 4: slots to the output; the masks cleared for the next tile
      const int rb = (int)(r + j0);
      for (int i = tid; i < total; i += kFillThreads) {
        const uint32_t rc = sRC[i];
        const typename VP::T v = sVal[i];
        const int dst = delta[rc >> 5] + i;
        row_out[dst] = rb + (int)(rc & 31u);
        DT[dst] = VP::d(v);
        LT[dst] = VP::l(v);
      }
      for (int k = tid; k < G / 4; k += kFillThreads) reinterpret_cast<uint4*>(mask)[k] = make_uint4(0u, 0u, 0u, 0u);
      __syncthreads();
      j0 = j1;
    }
  }
}

// The same transpose for rows with few entries per column group: then a tile of
// 32 rows holds too few entries for its passes over the group's columns, and the
// CTAs' look-ups of every (row, group) piece outgrow the entries.  One CTA takes
// the entries of strip b in CSR order, up to kScatEntries of up to 64 rows at a
// time, whatever their columns:
//   1  an entry finds its column's slot in a hash table (at most half full) and
//      sets its row's bit in the slot's 64-bit mask;
//   2  it goes to output cursor[c] + (its bits below its own): row order;
//   3  the first entry of a column advances the cursor and clears the slot.
// Entries of a tile rarely share a column, so every entry is a store of its own in
// each of the three arrays (4 sectors written per entry, most of them leaving L2 half
// empty; half of the stall cycles wait for the cursors): 12 to 15 ms per 1e8 entries
// whatever the shape.  Loads in ms, k_csc_fill (groups of 1024) -> k_csc_scatter, by mean
// entries per row and group:
//   9e-4 (9 per row, 3e6 columns, 1.8e7 entries)  184.8 -> 13.8   1.3   45.6 -> 27.7
//   0.1 (98, 1e6, 3.9e7)                          103.8 -> 11.9   2.5   23.8 -> 23.7
//   0.3 (19, 70000, 7.5e7)                         61.0 -> 15.0   3.3   27.0 -> 28.0
//   0.6 (19, 30000, 7.5e7)                         37.7 -> 15.0   6.6    6.1 -> 11.3
// Rows whose entries lie in a few of the groups favour k_csc_fill, so the line is 2.
// More than 65536 columns take one strip per SM, not two (their counters are 4
// bytes per strip and column): 17.8 -> 13.8 ms for 3e6 columns.
constexpr int kScatThreads = 512, kScatPer = 8, kScatEntries = kScatThreads * kScatPer;
constexpr int kScatSlotBits = 13, kScatSlots = 1 << kScatSlotBits;
constexpr int kScatRows = 1024;  // row pointers staged at a time
constexpr size_t kScatSmem = kScatSlots * (sizeof(unsigned long long) + sizeof(int32_t)) + (kScatRows + 1) * sizeof(int64_t);
static_assert(2 * kScatEntries <= kScatSlots, "hash table at most half full: every probe ends");

template <typename VT, typename IT>
__global__ void __launch_bounds__(kScatThreads, 2) k_csc_scatter(
    const int64_t* __restrict__ rp, const IT* __restrict__ col, const VT* __restrict__ Dv, const VT* __restrict__ Lv,
    const int64_t* __restrict__ strip_row, int32_t n_cols, int32_t* cursor, int32_t* __restrict__ row_out,
    VT* __restrict__ DT, VT* __restrict__ LT) {
  extern __shared__ __align__(16) unsigned char fill_sh[];
  unsigned long long* mask = reinterpret_cast<unsigned long long*>(fill_sh);
  int64_t* srp = reinterpret_cast<int64_t*>(mask + kScatSlots);
  int32_t* key = reinterpret_cast<int32_t*>(srp + kScatRows + 1);
  const int tid = threadIdx.x;
  for (int j = tid; j < kScatSlots; j += kScatThreads) {
    mask[j] = 0ull;
    key[j] = -1;
  }
  int32_t* cur = cursor + (int64_t)blockIdx.x * n_cols;
  const int64_t r_end = strip_row[blockIdx.x + 1];
  for (int64_t r0 = strip_row[blockIdx.x]; r0 < r_end; r0 += kScatRows) {
    const int nr = (int)min((int64_t)kScatRows, r_end - r0);
    for (int i = tid; i <= nr; i += kScatThreads) srp[i] = rp[r0 + i];
    __syncthreads();
    int64_t p0 = srp[0];
    for (int a = 0; a < nr;) {  // the tile starts at entry p0, in row a of the staged ones
      const int z = min(a + 64, nr);
      const int64_t p1 = min(p0 + kScatEntries, srp[z]);
      int c[kScatPer], hk[kScatPer];  // column or -1; slot | row of the tile << kScatSlotBits
#pragma unroll
      for (int q = 0; q < kScatPer; ++q) {
        const int64_t p = p0 + tid + q * kScatThreads;
        c[q] = p < p1 ? (int)col[p] : -1;
      }
#pragma unroll
      for (int q = 0; q < kScatPer; ++q) {
        if (c[q] < 0) continue;
        const int64_t p = p0 + tid + q * kScatThreads;
        int lo = a, hi = z;  // the last row that starts at or before p
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (srp[mid] <= p) lo = mid;
          else hi = mid;
        }
        unsigned h = ((unsigned)c[q] * 2654435761u) >> (32 - kScatSlotBits);
        while (true) {
          const int32_t k = atomicCAS(&key[h], -1, c[q]);
          if (k == -1 || k == c[q]) break;
          h = (h + 1) & (kScatSlots - 1);
        }
        atomicOr(&mask[h], 1ull << (lo - a));
        hk[q] = (int)h | ((lo - a) << kScatSlotBits);
      }
      __syncthreads();
      int next[kScatPer];  // the column's new cursor, where this entry is its first
#pragma unroll
      for (int q = 0; q < kScatPer; ++q) {
        next[q] = -1;
        if (c[q] < 0) continue;
        const int64_t p = p0 + tid + q * kScatThreads;
        const unsigned long long m = mask[hk[q] & (kScatSlots - 1)];
        const int row = hk[q] >> kScatSlotBits;
        const int rank = __popcll(m & ((1ull << row) - 1ull));
        const int base = cur[c[q]], pos = base + rank;
        row_out[pos] = (int)(r0 + a + row);
        DT[pos] = Dv[p];
        LT[pos] = Lv[p];
        if (rank == 0) next[q] = base + __popcll(m);
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kScatPer; ++q) {
        if (next[q] < 0) continue;
        const int h = hk[q] & (kScatSlots - 1);
        cur[c[q]] = next[q];
        key[h] = -1;
        mask[h] = 0ull;
      }
      if (p1 == srp[z]) {
        a = z;
      } else {  // the tile ended inside a row, or where one starts
        int hi = z;
        while (hi - a > 1) {
          const int mid = (a + hi) >> 1;
          if (srp[mid] <= p1) a = mid;
          else hi = mid;
        }
      }
      p0 = p1;
      __syncthreads();
    }
  }
}

template <typename VT, typename IT>
void scatter_inst(const CscShape& q, const int64_t* rp, const IT* col, const void* Dv, const void* Lv,
                  const int64_t* strip_row, int32_t* cursor, int32_t* row_out, void* DT, void* LT, cudaStream_t s) {
  k_csc_scatter<VT, IT><<<(unsigned)q.n_strip, kScatThreads, kScatSmem, s>>>(
      rp, col, (const VT*)Dv, (const VT*)Lv, strip_row, q.n_cols, cursor, row_out, (VT*)DT, (VT*)LT);
}

template <typename VT, typename IT>
void fill_inst(const CscShape& q, const int64_t* rp, const IT* col, const void* Dv, const void* Lv,
               const int64_t* strip_row, const int32_t* split, const int32_t* cursor, int32_t* row_out, void* DT,
               void* LT, cudaStream_t s) {
  const FillSmem<VT> m(q.tile, 1 << q.gshift);
  k_csc_fill<VT, IT><<<(unsigned)(q.n_strip * q.n_grp), kFillThreads, m.bytes, s>>>(
      rp, col, (const VT*)Dv, (const VT*)Lv, strip_row, q.n_strip, q.n_cols, q.gshift, q.n_grp, q.tile, split, cursor,
      row_out, (VT*)DT, (VT*)LT);
}

template <typename IT>
void count_inst(const CscShape& q, size_t smem_limit, const int64_t* rp, const IT* col, const int64_t* strip_row,
                int32_t* cnt, int32_t* split, cudaStream_t s) {
  const size_t smem = (size_t)q.n_cols * sizeof(int32_t);
  if (smem <= smem_limit) {
    k_csc_count<true, IT><<<q.n_strip, kCountThreads, smem, s>>>(rp, col, strip_row, q.n_cols, q.gshift, q.n_grp, cnt,
                                                                 split);
  } else {
    k_csc_count<false, IT><<<q.n_strip, kCountThreads, 0, s>>>(rp, col, strip_row, q.n_cols, q.gshift, q.n_grp, cnt,
                                                               split);
  }
}

// ------------------------------------------------------------------ columns, chunks, tiles

// Column pointers cp[0 .. n] from the column totals, and with chunks of C
// nonzeros the first chunk of every column (col_chunk[0 .. n]).  One block.
__global__ void __launch_bounds__(1024) k_csc_columns(const int64_t* __restrict__ tot, int32_t n, int64_t C,
                                                      int64_t* __restrict__ cp, int32_t* __restrict__ col_chunk) {
  __shared__ unsigned long long wp[32], wc[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  unsigned long long run_p = 0, run_c = 0;
  for (int64_t j0 = 0; j0 < n; j0 += 4096) {
    const int64_t j = j0 + 4 * (int64_t)threadIdx.x;  // four consecutive columns per thread
    unsigned long long v[4], own = 0, ch = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = j + k < n ? (unsigned long long)tot[j + k] : 0ull;
      own += v[k];
      ch += (v[k] + C - 1) / C;
    }
    unsigned long long x = own, y = ch;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long a = __shfl_up_sync(kFull, x, o), b = __shfl_up_sync(kFull, y, o);
      if (lane >= o) {
        x += a;
        y += b;
      }
    }
    if (lane == 31) {
      wp[wid] = x;
      wc[wid] = y;
    }
    __syncthreads();
    unsigned long long p = run_p + x - own, c = run_c + y - ch;
    for (int w = 0; w < 32; ++w) {
      if (w < wid) {
        p += wp[w];
        c += wc[w];
      }
      run_p += wp[w];
      run_c += wc[w];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (j + k < n) {
        cp[j + k] = (int64_t)p;
        col_chunk[j + k] = (int32_t)c;
      }
      p += v[k];
      c += (v[k] + C - 1) / C;
    }
    __syncthreads();  // wp and wc are rewritten
  }
  if (threadIdx.x == 0) {
    cp[n] = (int64_t)run_p;
    col_chunk[n] = (int32_t)run_c;
  }
}

// chunk_ptr: the chunks' first positions, column by column; then the end.
__global__ void k_chunk_fill(const int64_t* __restrict__ cp, const int32_t* __restrict__ col_chunk, int32_t n, int64_t C,
                             int64_t* __restrict__ chunk_ptr) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j == 0) chunk_ptr[col_chunk[n]] = cp[n];
  if (j >= n) return;
  const int64_t p0 = cp[j];
  const int c0 = col_chunk[j], c1 = col_chunk[j + 1];
  for (int c = c0; c < c1; ++c) chunk_ptr[c] = p0 + (int64_t)(c - c0) * C;
}

// First m in [a, z) whose prefix cost ptr[m] - ptr[a] + cost (m - a) reaches the target; z if none.
__device__ __forceinline__ int64_t find_cost(const int64_t* __restrict__ ptr, int64_t a, int64_t z, int64_t cost,
                                             double target) {
  const int64_t p0 = ptr[a];
  int64_t x = a, y = z;
  while (x < y) {
    const int64_t m = (x + y) / 2;
    if ((double)(ptr[m] - p0) + (double)cost * (double)(m - a) < target) x = m + 1;
    else y = m;
  }
  return x;
}

// Bound k of the split of one range [a, z) into `parts` pieces of equal cost.
__device__ __forceinline__ int64_t even_bound(const int64_t* ptr, int64_t a, int64_t z, int64_t cost, int k, int parts) {
  if (k <= 0) return a;
  if (k >= parts) return z;
  const double total = (double)(ptr[z] - ptr[a]) + (double)cost * (double)(z - a);
  return find_cost(ptr, a, z, cost, total * k / parts);
}

// Bound k of the guided tiles of [a, z) for W warps: W tiles of 1/2 of a warp's
// share, W of 1/4, 1/8, 1/16 and 1/32 each, 2 W of 1/64.
__device__ __forceinline__ int64_t guided_bound(const int64_t* ptr, int64_t a, int64_t z, int W, int64_t cost, int k) {
  if (k <= 0) return a;
  if (k >= kGuidedTilesPerWarp * W) return z;
  const double share = ((double)(ptr[z] - ptr[a]) + (double)cost * (double)(z - a)) / W;
  double done = 0.0, f = 0.5;
  int left = k;
  for (int round = 0; round < 5 && left > 0; ++round, f *= 0.5) {
    const int t = left < W ? left : W;
    done += f * t;
    left -= t;
  }
  done += 0.015625 * left;
  return find_cost(ptr, a, z, cost, done * share);
}

__global__ void k_tiles(TileArgs q) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (q.kind == TileArgs::PAIRS) {  // [r0, r1) of tile t: parts0 tiles over [a0, z0), then parts1 over [a1, z1)
    if (t >= q.parts0 + q.parts1) return;
    const bool second = t >= q.parts0;
    const int64_t a = second ? q.a1 : q.a0, z = second ? q.z1 : q.z0;
    const int k = second ? t - q.parts0 : t, parts = second ? q.parts1 : q.parts0;
    q.out64[2 * t] = even_bound(q.ptr, a, z, q.cost, k, parts);
    q.out64[2 * t + 1] = even_bound(q.ptr, a, z, q.cost, k + 1, parts);
  } else if (q.kind == TileArgs::BOUNDS64) {
    if (t <= q.parts0) q.out64[t] = even_bound(q.ptr, q.a0, q.z0, q.cost, t, q.parts0);
  } else if (q.kind == TileArgs::BOUNDS32) {
    if (t <= q.parts0) q.out32[t] = (int32_t)even_bound(q.ptr, q.a0, q.z0, q.cost, t, q.parts0);
  } else if (q.kind == TileArgs::GUIDED_PAIRS) {
    if (t >= kGuidedTilesPerWarp * q.parts0) return;
    q.out64[2 * t] = guided_bound(q.ptr, q.a0, q.z0, q.parts0, q.cost, t);
    q.out64[2 * t + 1] = guided_bound(q.ptr, q.a0, q.z0, q.parts0, q.cost, t + 1);
  } else {  // GUIDED32
    if (t <= kGuidedTilesPerWarp * q.parts0) q.out32[t] = (int32_t)guided_bound(q.ptr, q.a0, q.z0, q.parts0, q.cost, t);
  }
}

}  // namespace

// Groups of 1024 columns and kFillCtas CTAs per SM.  The tile takes the shared
// memory that is left; a slot's position fits 16 bits.
constexpr double kShortPiece = 2.0;  // mean entries per row and group below which k_csc_scatter takes over
CscShape csc_shape(const Geometry& g, int fmt, int64_t n_rows, int32_t n_cols, int64_t nnz) {
  CscShape q{};
  q.n_rows = n_rows;
  q.n_cols = n_cols;
  q.gshift = kFillGroupShift;
  while (q.gshift > 6 && (1 << (q.gshift - 1)) >= n_cols) --q.gshift;
  const int G = 1 << q.gshift;
  q.n_grp = (int)(((int64_t)n_cols + G - 1) >> q.gshift);
  q.short_pieces = (double)nnz < kShortPiece * (double)n_rows * (double)q.n_grp;
  q.n_strip = (int)std::max<int64_t>(1, std::min<int64_t>((int64_t)g.n_sms * (q.short_pieces && n_cols > 65536 ? 1 : 2), n_rows));
  const size_t budget = (g.smem_limit - 1024 * (kFillCtas - 1)) / kFillCtas;
  const int per = fmt == 0 ? 12 : 8;
  const size_t fixed = fmt == 0 ? FillSmem<float>(0, G).bytes : FillSmem<uint16_t>(0, G).bytes;
  q.tile = (int)std::min<size_t>(16384, (budget - fixed - 64) / per) & ~15;
  // the table of the groups' starts pays when it stays below the matrix itself
  q.use_split = !q.short_pieces && (double)(q.n_grp + 1) * 4.0 * (double)n_rows <= 8.0 * (double)nnz;
  return q;
}

void launch_csc_count(const CscShape& q, size_t smem_limit, const int64_t* rp, const int32_t* col,
                      const uint16_t* col16, const int64_t* strip_row, int32_t* cnt, int32_t* split, cudaStream_t s) {
  if (col16) count_inst(q, smem_limit, rp, col16, strip_row, cnt, split, s);
  else count_inst(q, smem_limit, rp, col, strip_row, cnt, split, s);
}

void launch_csc_colsum(const int32_t* cnt, int n_strip, int32_t n_cols, int64_t* tot, cudaStream_t s) {
  k_csc_colsum<<<(n_cols + 255) / 256, 256, 0, s>>>(cnt, n_strip, n_cols, tot);
}

void launch_csc_offsets(int32_t* cnt, int n_strip, int32_t n_cols, const int64_t* cp, cudaStream_t s) {
  k_csc_offsets<<<(n_cols + 255) / 256, 256, 0, s>>>(cnt, n_strip, n_cols, cp);
}

void launch_csc_fill(const CscShape& q, int fmt, const int64_t* rp, const int32_t* col, const uint16_t* col16,
                     const void* Dv, const void* Lv, const int64_t* strip_row, const int32_t* split,
                     int32_t* cursor, int32_t* row_out, void* DT, void* LT, cudaStream_t s) {
  auto go = [&](auto v, auto cols) {
    using VT = decltype(v);
    if (q.short_pieces) scatter_inst<VT>(q, rp, cols, Dv, Lv, strip_row, cursor, row_out, DT, LT, s);
    else fill_inst<VT>(q, rp, cols, Dv, Lv, strip_row, split, cursor, row_out, DT, LT, s);
  };
  if (fmt == 0 && col16) go(float(), col16);
  else if (fmt == 0) go(float(), col);
  else if (col16) go(uint16_t(), col16);
  else go(uint16_t(), col);
}

void launch_csc_columns(const int64_t* tot, int32_t n, int64_t C, int64_t* cp, int32_t* col_chunk, cudaStream_t s) {
  k_csc_columns<<<1, 1024, 0, s>>>(tot, n, C, cp, col_chunk);
}

void launch_chunk_fill(const int64_t* cp, const int32_t* col_chunk, int32_t n, int64_t C, int64_t* chunk_ptr,
                       cudaStream_t s) {
  k_chunk_fill<<<(unsigned)(((int64_t)n + 255) / 256), 256, 0, s>>>(cp, col_chunk, n, C, chunk_ptr);
}

void launch_tiles(const TileArgs& q, cudaStream_t s) {
  const int64_t t = q.kind == TileArgs::PAIRS            ? (int64_t)q.parts0 + q.parts1
                    : q.kind == TileArgs::GUIDED_PAIRS || q.kind == TileArgs::GUIDED32
                        ? (int64_t)kGuidedTilesPerWarp * q.parts0 + 1
                        : (int64_t)q.parts0 + 1;
  k_tiles<<<(unsigned)((t + 127) / 128), 128, 0, s>>>(q);
}

int64_t row_order_blocks(int64_t n_rows) { return std::max<int64_t>(1, (n_rows + kRowBlk - 1) / kRowBlk); }
size_t row_order_scratch(int64_t n_rows) { return (size_t)row_order_blocks(n_rows) * kRowCounters; }

void launch_rows_count(const int64_t* rp, const uint32_t* mask, int64_t n, int64_t nnz, bool roi, int64_t* blk,
                       RowTotals* tot, cudaStream_t s) {
  const int64_t nb = row_order_blocks(n);
  k_rows_count<<<(unsigned)nb, 256, 0, s>>>(rp, mask, n, nnz, roi ? 1 : 0, blk, tot);
  k_rows_scan<<<1, kRowCounters * 32, 0, s>>>(blk, nb, tot);
}

void launch_rows_place(const int64_t* rp, const uint32_t* mask, int64_t n, bool roi, const int64_t* blk,
                       const RowTotals* tot, int64_t* rp_out, int64_t* voxel, uint32_t* mask_out, int64_t* con_rows,
                       float* sD, float* sL, cudaStream_t s) {
  k_rows_place<<<(unsigned)row_order_blocks(n), 256, 0, s>>>(rp, mask, n, roi ? 1 : 0, blk, tot, rp_out, voxel,
                                                             mask_out, con_rows, sD, sL);
}

template <typename IT>
static cudaError_t init_load_it(int bytes) {
  const void* k[] = {(const void*)k_csc_count<true, IT>,       (const void*)k_csc_fill<float, IT>,
                     (const void*)k_csc_fill<uint16_t, IT>,    (const void*)k_csc_scatter<float, IT>,
                     (const void*)k_csc_scatter<uint16_t, IT>};
  for (const void* f : k) {
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t init_load_kernels(int smem_bytes) {
  const cudaError_t e = init_load_it<int32_t>(smem_bytes);
  return e != cudaSuccess ? e : init_load_it<uint16_t>(smem_bytes);
}

template <typename VT, bool COPY>
static void load_rows_inst(const LoadRowsArgs& a, bool narrow, unsigned grid, cudaStream_t s) {
  if (narrow) k_load_rows<VT, uint16_t, COPY><<<grid, 256, 0, s>>>(a);
  else k_load_rows<VT, int32_t, COPY><<<grid, 256, 0, s>>>(a);
}

void launch_load_rows(int fmt, bool narrow, bool copy_values, const LoadRowsArgs& a, cudaStream_t s) {
  const int64_t jobs = a.n_hot_ne + a.n_cold_ne;
  if (jobs == 0) return;
  const unsigned grid = (unsigned)std::min<int64_t>((jobs + 7) / 8, 65535);
  if (fmt == 1) load_rows_inst<__nv_bfloat16, true>(a, narrow, grid, s);
  else if (fmt == 2) load_rows_inst<__half, true>(a, narrow, grid, s);
  else if (copy_values) load_rows_inst<float, true>(a, narrow, grid, s);
  else load_rows_inst<float, false>(a, narrow, grid, s);
}

}  // namespace fo
