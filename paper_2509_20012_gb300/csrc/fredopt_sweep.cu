// The block-iterative sweep: the block form of Fig. 2's row-action sweep.
// Per block of structure rows, three kernels chained by programmatic dependent
// launch:
//   k_sweep_rows  forward product of the block's rows, several warps per row
//                 (blocks of many nonzeros or many short rows: k_forward)
//   k_sweep_con   half-space evaluation, one row per thread
//   k_sweep_cols  x_j += scale * sum over the block's entries of column j
// A block of the clinical plan holds a few hundred rows (9 MB of matrix), so a
// block is a chain of latencies, not of bytes: every kernel loads what does not
// depend on its predecessor (matrix entries, positions, moments) before it waits
// for it, and a row or column is spread over as many lanes as its length fills.
// Clinical plan (5.7e7 nonzeros in structure rows, FP32), one sweep: 64 blocks
// 3.60 -> 1.21 ms against plain launches of the streaming forward kernel (one
// warp per row), the constraint kernel over 608 CTAs and one warp per column;
// 1 block 0.44 -> 0.28 ms.  The chain is kept in batches too, where it was
// measured: six plans of 64 blocks 1.77 -> 0.76 ms per iteration.
#include "fredopt.h"
#include "fredopt_device.cuh"
#include "fredopt_internal.cuh"

#include <algorithm>

namespace fo {

namespace {

// x = w + coef * g (the perturbed point; coef = 0 without perturbation), and
// the sweep's violation counters cleared.
__global__ void k_sweep_start(int n, const float* __restrict__ w, const float* __restrict__ g, int use_coef,
                              float* __restrict__ x, DevState* st) {
  const double coef = use_coef ? st->coef : 0.0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    x[j] = use_coef ? (float)((double)w[j] + coef * (double)g[j]) : w[j];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    st->sweep_nv = 0ull;
    st->sweep_mx = 0ll;
  }
}

// pos[t * n + j] = first CSC position of column j whose row is >= bounds[t].
__global__ void k_sweep_pos(const int64_t* __restrict__ cp, const int32_t* __restrict__ row, int32_t n,
                            const int64_t* __restrict__ bounds, int n_bounds, int64_t* __restrict__ pos) {
  const int64_t total = (int64_t)n_bounds * n;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (int64_t)gridDim.x * blockDim.x) {
    const int t = (int)(idx / n);
    const int j = (int)(idx - (int64_t)t * n);
    const int64_t target = bounds[t];
    int64_t lo = cp[j], hi = cp[j + 1];
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if ((int64_t)row[mid] < target) lo = mid + 1;
      else hi = mid;
    }
    pos[idx] = lo;
  }
}

// Per block, over its columns: out[2 t] = entries, out[2 t + 1] = sum of their squares
// (their ratio is the length of the column that an entry lies in, on average).
__global__ void __launch_bounds__(256) k_sweep_lengths(const int64_t* __restrict__ pos, int32_t n, double* out) {
  __shared__ double red[9];
  const int64_t* p = pos + (int64_t)blockIdx.x * n;
  double s1 = 0.0, s2 = 0.0;
  for (int j = threadIdx.x; j < n; j += 256) {
    const double l = (double)(p[n + j] - p[j]);
    s1 += l;
    s2 += l * l;
  }
  s1 = block_sum256(s1, red);
  s2 = block_sum256(s2, red);
  if (threadIdx.x == 0) {
    out[2 * blockIdx.x] = s1;
    out[2 * blockIdx.x + 1] = s2;
  }
}

// Priority sum of the reachable constraint rows of slice blockIdx.y of block
// blockIdx.x (`rows` rows).  One CTA over a whole block of 79 thousand rows took
// 0.46 ms.
__global__ void __launch_bounds__(256) k_sweep_weights(Tables t, const int64_t* list, int64_t n_list, int64_t size,
                                                       int64_t rows, const uint32_t* mask, const double* dd,
                                                       const double* ll, const double* dl, double* part) {
  __shared__ double red[9];
  const int64_t b0 = (int64_t)blockIdx.x * size, b1 = min(n_list, b0 + size);
  const int64_t i0 = b0 + (int64_t)blockIdx.y * rows, i1 = min(b1, i0 + rows);
  double p = 0.0;
  for (int64_t i = i0 + threadIdx.x; i < i1; i += 256) {
    const int64_t r = list[i];
    const uint32_t m = mask[r];
    for (int q = 0; q < t.n_con; ++q)
      if (((m >> t.con[q].bit) & 1u) && row_norm2(t.con[q], t.c, dd[r], ll[r], dl[r]) > 0.0) p += t.con[q].prio;
  }
  p = block_sum256(p, red);
  if (threadIdx.x == 0) part[(int64_t)blockIdx.x * gridDim.y + blockIdx.y] = p;
}

__global__ void __launch_bounds__(256) k_sweep_winv(const double* part, int slices, double* winv) {
  __shared__ double red[9];
  const double p = block_sum_array(part + (int64_t)blockIdx.x * slices, slices, red);
  if (threadIdx.x == 0) winv[blockIdx.x] = p > 0.0 ? 1.0 / p : 0.0;
}

// (Dx, Lx) of the block's rows, WPR warps per row: a lane takes every
// (32 WPR)-th entry, four of them in flight, the next four requested before
// the current ones are used.
template <typename VT, typename IT, int WPR>
__global__ void __launch_bounds__(256) k_sweep_rows(SweepArgs a) {
  constexpr int K = 4, GS = 32 * WPR;
  __shared__ float2 part[8];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t i = a.i0 + (int64_t)blockIdx.x * (8 / WPR) + wid / WPR;
  const bool have = i < a.i1;
  const int64_t r = have ? checked_index(a.list[i], a.n_rows, a.st) : 0;
  const int64_t s = have ? a.rp[r] : 0;
  const int len = have ? (int)(checked_end(s, a.rp[r + 1], a.n_elems, a.st) - s) : 0;
  const IT* __restrict__ ci = (sizeof(IT) == 2 ? reinterpret_cast<const IT*>(a.col16) : reinterpret_cast<const IT*>(a.col)) + s;
  const VT* __restrict__ Di = reinterpret_cast<const VT*>(a.rD) + s;
  const VT* __restrict__ Li = reinterpret_cast<const VT*>(a.rL) + s;
  const int first = (wid % WPR) * 32 + lane;
  int c[K];
  VT d[K], l[K];
  auto load = [&](int e0) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int e = e0 + k * GS;
      c[k] = -1;
      if (e < len) {
        c[k] = (int)ci[e];
        d[k] = Di[e];
        l[k] = Li[e];
      }
    }
  };
  load(first);
  pdl_wait();  // x is the last block's
  pdl_release();
  float sA = 0.0f, sB = 0.0f;
  for (int e0 = first; __any_sync(kFull, e0 < len); e0 += K * GS) {
    float x[K], dv[K], lv[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      x[k] = c[k] >= 0 ? a.x[checked_index(c[k], a.n, a.st)] : 0.0f;
      dv[k] = c[k] >= 0 ? to_f(d[k]) : 0.0f;
      lv[k] = c[k] >= 0 ? to_f(l[k]) : 0.0f;
    }
    load(e0 + K * GS);
#pragma unroll
    for (int k = 0; k < K; ++k) {
      sA = fmaf(dv[k], x[k], sA);
      sB = fmaf(lv[k], x[k], sB);
    }
  }
  warp_sum2(sA, sB, lane);
  if (WPR > 1) {
    if (lane == 0) part[wid] = make_float2(sA, sB);
    __syncthreads();
  }
  if (have && first == 0) {
    if (WPR > 1) {
#pragma unroll
      for (int k = 1; k < WPR; ++k) {
        sA += part[wid + k].x;
        sB += part[wid + k].y;
      }
    }
    // row scales are powers of two: the FP32 product is exact
    a.y[r] = a.sD ? make_float2(sA * a.sD[r], sB * a.sL[r]) : make_float2(sA, sB);
  }
}

// One row per thread, one warp per CTA: the FP64 divisions spread over the SMs.
__global__ void __launch_bounds__(kSweepConThreads) k_sweep_con(SweepArgs a, Tables t) {
  __shared__ ConEntry con[kMaxCon];
  stage_constraints(t, con);
  const int64_t i = a.i0 + (int64_t)blockIdx.x * kSweepConThreads + threadIdx.x;
  const bool have = i < a.i1;
  const int64_t r = have ? checked_index(a.list[i], a.n_rows, a.st) : 0;
  const uint32_t m = have ? a.mask[r] : 0u;
  const double dd = have ? a.dd[r] : 0.0, ll = have ? a.ll[r] : 0.0, dl = have ? a.dl[r] : 0.0;
  const double sd = have && a.sD ? (double)a.sD[r] : 1.0, sl = have && a.sL ? (double)a.sL[r] : 1.0;
  __syncthreads();
  const uint32_t todo = row_constraints(con, t.n_con, m);
  pdl_wait();  // y of this block
  pdl_release();
  const float2 y = have ? a.y[r] : make_float2(0.0f, 0.0f);
  double gD = 0.0, gL = 0.0, psum = 0.0, preach = 0.0, mx = 0.0;
  unsigned nv = 0u;
  eval_constraints(con, todo, t.c, y.x, y.y, dd, ll, dl, gD, gL, psum, preach, nv, mx);
  if (have) a.gam[r] = make_float2((float)(gD * sd), (float)(gL * sl));
  if (a.norm == FREDOPT_NORM_VIOLATED) {
    psum = warp_sum_nz(psum);
    if (threadIdx.x == 0) a.part[blockIdx.x] = psum;
  }
  if (a.in_solve) {  // exact whatever the order: integers, and a maximum of doubles >= 0 by their bits
    nv = __reduce_add_sync(kFull, nv);
    const long long bits = warp_max_bits(__double_as_longlong(mx));
    if (threadIdx.x == 0 && nv) {
      atomicAdd(&a.st->sweep_nv, (unsigned long long)nv);
      atomicMax(&a.st->sweep_mx, bits);
    }
  }
}

// x_j += lam * scale / W_B * sum over the block's entries of column j of
// D_ij gamma_D[i] + L_ij gamma_L[i].  LPC lanes per column, U columns per lane
// group, K entries of each in flight together: four of one long column, or one
// each of two short ones.  The FP64 update is left to the
// CTA's first warps, one column per lane: GB300 issues an FP64 warp instruction
// at the same low rate however few of its lanes are active, and one update per
// column in the column's own warp was most of this kernel's time (19 us per
// block of the clinical plan at 64 blocks).  A block's share of the columns is
// uneven (its rows lie at one place), which is what is left.
constexpr int kColsU = 2;  // columns per lane group (with 8 CTAs per SM: 3% faster than 4 with 4)
template <typename VT, int LPC, int U, int K, int CTAS>
__global__ void __launch_bounds__(256, CTAS) k_sweep_cols(SweepArgs a) {
  constexpr int CPW = 32 / LPC, COLS = 8 * U * CPW;  // columns per CTA
  __shared__ float sums[COLS];
  __shared__ double red[9];
  __shared__ double sh_scale;
  const int lane = threadIdx.x & 31;
  const int sl = lane % LPC;
  const int jw = (threadIdx.x >> 5) * (U * CPW) + lane / LPC;  // first column of the lane group, in the CTA
  const int64_t jc = (int64_t)blockIdx.x * COLS;  // (columns dealt out with the grid's stride: 12% slower)
  const VT* __restrict__ Dv = reinterpret_cast<const VT*>(a.Dv);
  const VT* __restrict__ Lv = reinterpret_cast<const VT*>(a.Lv);
  int p[U], left[U];  // positions are below 2^31
  int most = 0;
#pragma unroll
  for (int k = 0; k < U; ++k) {
    const int64_t j = jc + jw + k * CPW;
    const int64_t p0 = j < a.n ? a.pos0[j] : 0, p1 = j < a.n ? checked_end(p0, a.pos1[j], a.n_csc, a.st) : 0;
    p[k] = (int)p0 + sl;
    left[k] = (int)(p1 - p0) - sl;
    most = max(most, left[k]);
  }
  int row[U][K];
  VT d[U][K], l[U][K];
  auto load = [&](int o) {
#pragma unroll
    for (int k = 0; k < U; ++k) {
#pragma unroll
      for (int e = 0; e < K; ++e) {
        row[k][e] = -1;
        if (o + e * LPC < left[k]) {
          row[k][e] = a.row[p[k] + o + e * LPC];
          d[k][e] = Dv[p[k] + o + e * LPC];
          l[k][e] = Lv[p[k] + o + e * LPC];
        }
      }
    }
  };
  load(0);
  // the step: with NORM_ALL 1 / W_B is known before the predecessor ends
  auto step_of = [&](double winv) {
    if (threadIdx.x == 0) {
      const double ps = a.in_solve ? (a.st->eta == 1.0 ? 1.0 : pow(a.st->eta, (double)a.st->k)) : a.prio_scale;
      sh_scale = a.lam * ps * winv;
    }
  };
  if (a.norm != FREDOPT_NORM_VIOLATED) step_of(*a.winv);
  pdl_wait();  // gam (and the partial sums) of this block
  pdl_release();
  const int64_t jt = jc + threadIdx.x;
  const bool mine = threadIdx.x < COLS && jt < a.n;  // this thread updates x[jt]
  const float xj = mine ? a.x[jt] : 0.0f;
  if (a.norm == FREDOPT_NORM_VIOLATED) {
    double v = 0.0;
    for (int i = threadIdx.x; i < a.con_blocks; i += 256) v += a.part[i];
    v = block_sum256(v, red);
    step_of(v > 0.0 ? 1.0 / v : 0.0);
  }
  float acc[U];
#pragma unroll
  for (int k = 0; k < U; ++k) acc[k] = 0.0f;
  for (int o = 0; __any_sync(kFull, o < most); o += LPC * K) {
    float2 g[U][K];
    float dv[U][K], lv[U][K];
#pragma unroll
    for (int k = 0; k < U; ++k) {
#pragma unroll
      for (int e = 0; e < K; ++e) {
        g[k][e] = row[k][e] >= 0 ? a.gam[checked_index(row[k][e], a.n_rows, a.st)] : make_float2(0.0f, 0.0f);
        dv[k][e] = row[k][e] >= 0 ? to_f(d[k][e]) : 0.0f;
        lv[k][e] = row[k][e] >= 0 ? to_f(l[k][e]) : 0.0f;
      }
    }
    load(o + LPC * K);
#pragma unroll
    for (int k = 0; k < U; ++k) {
#pragma unroll
      for (int e = 0; e < K; ++e) {
        acc[k] = fmaf(dv[k][e], g[k][e].x, acc[k]);
        acc[k] = fmaf(lv[k][e], g[k][e].y, acc[k]);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < U; ++k) {
#pragma unroll
    for (int o = LPC / 2; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(kFull, acc[k], o);
    if (sl == 0) sums[jw + k * CPW] = acc[k];
  }
  __syncthreads();
  if (mine) {
    const float s = sums[threadIdx.x];
    if (s != 0.0f) a.x[jt] = (float)((double)xj + sh_scale * (double)s);
  }
}

// out = max(0, x); in a solve the last block writes the log entry and advances k.
__global__ void __launch_bounds__(256) k_sweep_finish(int n, const float* __restrict__ x, float* __restrict__ out,
                                                      int in_solve, DevState* st, LogEntry* log) {
  __shared__ bool sh_last;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x)
    out[j] = x[j] > 0.0f ? x[j] : 0.0f;
  if (!in_solve) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned prev = atomicAdd(&st->done, 1u);
    sh_last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (sh_last && threadIdx.x == 0) {
    __threadfence();
    if (st->log_cap > 0) {
      LogEntry e;
      e.k = st->k;
      e.s = st->s;
      e.accepted = st->accepted;
      e.n_violated = (int)st->sweep_nv;
      e.beta = st->beta_acc;
      e.f_start = st->f_start;
      e.f_end = st->f_cur;
      e.gnorm = st->gnorm;
      e.max_violation = __longlong_as_double(st->sweep_mx);
      log[st->k % st->log_cap] = e;
    }
    st->k += 1;
    st->done = 0u;
  }
}

template <typename VT, typename IT>
void rows_inst(double mean_nnz, const SweepArgs& a, cudaStream_t s) {
  const int64_t rows = a.i1 - a.i0;
  auto go = [&](auto kernel, int wpr) {
    launch_chain(true, kernel, (unsigned)((rows * wpr + 7) / 8), 256, 0, s, a);
  };
  if (mean_nnz >= 1024.0) go(k_sweep_rows<VT, IT, 8>, 8);
  else if (mean_nnz >= 512.0) go(k_sweep_rows<VT, IT, 4>, 4);
  else if (mean_nnz >= 192.0) go(k_sweep_rows<VT, IT, 2>, 2);
  else go(k_sweep_rows<VT, IT, 1>, 1);
}

template <typename VT>
void cols_inst(double mean_entries, double own_entries, const SweepArgs& a, cudaStream_t s) {
  auto go = [&](auto kernel, int cols) {
    launch_chain(true, kernel, (unsigned)(((int64_t)a.n + cols - 1) / cols), 256, 0, s, a);
  };
  // The update of one sweep, in us, two columns and one entry each in flight per
  // lane -> one column and four entries, by the entries of the column that an entry
  // lies in (a block's columns are uneven):
  //   30000 columns   161  993 -> 1136   318  602 -> 635   478  498 ->  399   865  803 -> 494   2028 3674 -> 2422
  //   70000           107  290 ->  351   425  228 -> 223        50000   333  269 ->  316   666  228 -> 229
  //   2000            142 1153 ->  854   440  662 -> 373   879  533 ->  260
  // Few columns are few warps either way; short ones share the GPU worse then (six
  // plans of 640 to 6480 columns in a batch: 77 to 185 entries 375 -> 400 us per
  // iteration, 224 to 575 290 -> 274).
  if (own_entries > (a.n < 8192 ? 200.0 : 400.0)) go(k_sweep_cols<VT, 32, 1, 4, 4>, 8);
  else if (mean_entries > 12.0) go(k_sweep_cols<VT, 32, kColsU, 1, 8>, 8 * kColsU);
  else go(k_sweep_cols<VT, 8, kColsU, 1, 8>, 8 * kColsU * 4);
}

}  // namespace

void launch_sweep_start(int n, const float* w, const float* g, int use_coef, float* x, DevState* st,
                        cudaStream_t s) {
  k_sweep_start<<<std::max(1, std::min(1024, (n + 255) / 256)), 256, 0, s>>>(n, w, g, use_coef, x, st);
}

void launch_sweep_pos(const int64_t* cp, const int32_t* row, int32_t n, const int64_t* bounds, int n_bounds,
                      int64_t* pos, cudaStream_t s) {
  const int64_t total = (int64_t)n_bounds * n;
  if (total == 0) return;
  const unsigned gb = (unsigned)std::min<int64_t>((total + 255) / 256, 65535);
  k_sweep_pos<<<gb, 256, 0, s>>>(cp, row, n, bounds, n_bounds, pos);
}

int sweep_weight_slices(int64_t size) {
  return (int)std::min<int64_t>(4096, std::max<int64_t>(1, (size + 1023) / 1024));
}

void launch_sweep_weights(const Tables& t, const int64_t* list, int64_t n_list, int64_t size, int n_blk,
                          const uint32_t* mask, const double* dd, const double* ll, const double* dl, double* part,
                          double* winv, cudaStream_t s) {
  if (n_blk == 0) return;
  const int slices = sweep_weight_slices(size);
  k_sweep_weights<<<dim3(n_blk, slices), 256, 0, s>>>(t, list, n_list, size, (size + slices - 1) / slices, mask, dd, ll, dl,
                                                      part);
  k_sweep_winv<<<n_blk, 256, 0, s>>>(part, slices, winv);
}

void launch_sweep_rows(int fmt, double mean_nnz, const SweepArgs& a, cudaStream_t s) {
  auto by_index = [&](auto v) {
    using VT = decltype(v);
    if (a.col16) rows_inst<VT, uint16_t>(mean_nnz, a, s);
    else rows_inst<VT, int32_t>(mean_nnz, a, s);
  };
  if (fmt == 1) by_index(__nv_bfloat16());
  else if (fmt == 2) by_index(__half());
  else by_index(float());
}

void launch_sweep_con(const Tables& t, const SweepArgs& a, cudaStream_t s) {
  launch_chain(true, k_sweep_con, (unsigned)a.con_blocks, kSweepConThreads, 0, s, a, t);
}

void launch_sweep_lengths(const int64_t* pos, int32_t n, int n_blk, double* out, cudaStream_t s) {
  if (n_blk > 0) k_sweep_lengths<<<n_blk, 256, 0, s>>>(pos, n, out);
}

void launch_sweep_cols(int fmt, double mean_entries, double own_entries, const SweepArgs& a, cudaStream_t s) {
  if (fmt == 1) cols_inst<__nv_bfloat16>(mean_entries, own_entries, a, s);
  else if (fmt == 2) cols_inst<__half>(mean_entries, own_entries, a, s);
  else cols_inst<float>(mean_entries, own_entries, a, s);
}

void launch_sweep_finish(const Geometry& g, int n, const float* x, float* out, int in_solve, DevState* st,
                         LogEntry* log, cudaStream_t s) {
  const unsigned gb = (unsigned)std::max(1, std::min(g.n_sms, (n + 255) / 256));
  k_sweep_finish<<<gb, 256, 0, s>>>(n, x, out, in_solve, st, log);
}

}  // namespace fo
