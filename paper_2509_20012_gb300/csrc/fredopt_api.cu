// C ABI of libfredopt (include/fredopt.h): plan upload and setup (stage
// (iii) of Table 2), the device-resident iteration of Fig. 3 around the
// simultaneous form of Fig. 2, and the final FP64 outputs.
//
// Device order of rows: with FREDOPT_ROWS_ROI the rows of voxels that belong
// to some structure come first (ascending voxel), then all other rows; the
// iteration streams only the first n_hot rows (Fig. 2 visits the voxels of
// the ROIs only).  With FREDOPT_ROWS_ALL the order is the voxel order and
// every row is streamed every pass.  The final outputs always cover every
// voxel.
#include "fredopt.h"
#include "fredopt_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <memory>
#include <string>
#include <vector>

using namespace fo;

namespace {

template <typename T>
struct DBuf {
  T* p = nullptr;
  size_t n = 0;
  DBuf() = default;
  DBuf(const DBuf&) = delete;
  DBuf& operator=(const DBuf&) = delete;
  ~DBuf() { release(); }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    n = 0;
  }
  cudaError_t alloc(size_t count) {
    release();
    const size_t c = count ? count : 1;
    cudaError_t e = cudaMalloc(reinterpret_cast<void**>(&p), c * sizeof(T));
    if (e == cudaSuccess) n = count;
    else p = nullptr;
    return e;
  }
  cudaError_t ensure(size_t count) { return (p && n >= count) ? cudaSuccess : alloc(count); }
  // a reload keeps a buffer that is large enough and at most twice as large
  cudaError_t fit(size_t count) { return (p && n >= count && n / 2 <= count) ? cudaSuccess : alloc(count); }
};

struct Timer {
  cudaEvent_t a = nullptr, b = nullptr;
  int cls = 0;
};

// the two event-record nodes around one kernel of a timed iteration graph
struct GraphTimer {
  cudaGraphNode_t a = nullptr, b = nullptr;
  int cls = 0;
};

// Blocks of the block-iterative sweep (built for m requested blocks; 0 = not built)
struct Sweep {
  int m = 0;
  int nb = 0;                      // blocks actually formed
  int64_t size = 0;                // structure rows with nonzeros per block
  int warps = 0;                   // > 0: the streaming forward product takes the blocks' rows,
  DBuf<int64_t> tiles;             // in this many tiles per block
  DBuf<int64_t> pos, bounds;
  DBuf<double> lens;               // scratch of the build
  double own_entries = 0.0;        // entries of a block in the column that an entry lies in, on average
  DBuf<double> w, wpart;           // [nb] 1 / priority sum; its slices' sums
  DBuf<double> part;               // violated rows' partial priority sums of a block
};

}  // namespace

struct fredopt_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  bool own_stream = false;
  cudaEvent_t ev_join = nullptr, ev_it0 = nullptr, ev_it1 = nullptr;
  Geometry geo{};       // launch shapes of the loaded plan
  Geometry geo_full{};  // the device's full-GPU shapes
  std::string last_error;
  size_t l2_bytes = 0;

  // plan
  bool loaded = false;
  int fmt = 0;
  bool roi = false;
  int64_t V = 0, nnz = 0, n_hot = 0, nnz_hot = 0;
  int64_t n_hot_ne = 0, n_cold_ne = 0;  // rows with nonzeros among streamed / other rows
  bool perm = false;                    // device order differs from voxel order
  int32_t n = 0, n_pad = 0;
  DBuf<int64_t> rp;
  DBuf<int32_t> col;
  DBuf<uint16_t> col16;  // 16-bit copy of col for the forward stream (col then freed)
  DBuf<uint8_t> Dv, Lv;
  DBuf<float> sD, sL;
  DBuf<int64_t> voxel;  // device row -> voxel (when perm)
  DBuf<uint32_t> mask;  // [n_hot]
  DBuf<double> mdd, mll, mdl;
  DBuf<int64_t> cp;
  DBuf<int32_t> crow;
  // based 16-bit copy of crow for the transposed product (per 128-element
  // block: base row in chdr, or an overflow slot of covf for wide blocks)
  DBuf<uint16_t> crow16;
  DBuf<int32_t> chdr, covf;
  DBuf<unsigned int> cnw;
  int64_t n_wide_blocks = 0;
  DBuf<uint8_t> DTv, LTv;
  DBuf<int64_t> warp_row_hot, warp_row_all, chunk_ptr;
  DBuf<int64_t> tile_row_hot;  // claimed tiles of the streamed rows (guided sizes)
  int n_tiles_hot = 0;
  DBuf<int64_t> tile_row_all;  // the same for every row with nonzeros, whole-GPU shapes
  int n_tiles_all = 0;
  DBuf<unsigned int> fsched;   // counters of the claimed tiles
  DBuf<int32_t> tile_chunk;    // claimed tiles of the transposed product: chunk bounds [n_tiles_bwd + 1]
  int n_tiles_bwd = 0;
  DBuf<unsigned int> bsched;
  DBuf<int32_t> col_chunk, warp_chunk;
  int64_t n_chunks = 0;
  bool hint_fwd = true, hint_bwd = true;
  int64_t row_cost = 0, chunk_cost = 0;  // warp-partition weights in use
  DBuf<int64_t> con_rows;        // streamed rows with a structure bit, ascending
  int64_t n_con_rows = 0, n_con_ne = 0;  // all of them; those with nonzeros (first in the list)
  int64_t con_nnz = 0;                   // nonzeros of the structure rows
  uint64_t empty_bits[32] = {0};  // streamed rows without nonzeros, per structure bit
  DBuf<float2> ucoef;            // coefficients of fredopt_backward (kept apart from gam)

  // problem
  Tables tab{};
  bool have_con = false;
  bool obj_dose = false;
  double W_all = 0.0;
  int64_t n_rows_reach = 0, n_unreach = 0;

  // buffers
  DBuf<float> w, g, xbuf, gtmp;
  DBuf<float2> yw, yg, r, gam, yall;
  DBuf<double2> y64;
  // y64 / yall were zeroed since the load: the products write rows with
  // nonzeros only, so the other rows stay 0
  bool y64_zeroed = false, yall_zeroed = false;
  DBuf<float> chunk_sum, fout_a, fout_b, vin_a, vin_b;
  DBuf<uint8_t> vol_buf;  // volume statistics scratch

  std::unique_ptr<Sweep> sw{new Sweep()};    // blocks of the begun solve's sweeps, or of the last single sweep
  DBuf<float> xs;                            // the point being swept [n_pad]
  DBuf<float2> ys;                           // forward product of a block's rows [n_con_ne]
  DBuf<double> part;
  // steps beta0 alpha^s of the trial loop for s < kBetaTable (in `part` at
  // off_btab), filled on the device for (btab_alpha, btab_beta0)
  double btab_alpha = -1.0, btab_beta0 = -1.0;
  DBuf<DevState> st;
  DBuf<LogEntry> log;
  DBuf<int> errw;
  // pinned host memory: the error word that kernels set (mapped), and a staging
  // area for the small results a call returns with
  uint8_t* pin = nullptr;
  int* err_dev = nullptr;  // device address of the error word
  size_t off_f = 0, off_bc = 0, off_g = 0, off_k2 = 0, off_fin = 0, off_cnt = 0, off_stage = 0, off_btab = 0,
         n_part = 0;

  // solve
  bool begun = false;
  fredopt_params prm{};
  double alpha = 0.99, lam = 1.0, beta0 = 0.0;
  int64_t iters_run = 0;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t gexec = nullptr;
  int graph_nodes = 0;
  double device_ms = 0.0;
  bool it_pending = false;
  DevState st_host{};

  // timing
  bool timing = false;
  std::vector<Timer> timers;
  size_t timers_used = 0;
  bool capturing = false;            // enqueue_iteration is being captured into `graph`
  bool graph_timed = false;          // `graph` holds an event pair around each kernel
  std::vector<GraphTimer> gtimers;   // those pairs, in kernel order
  double kms[FREDOPT_KCLASS_N] = {0};
  int64_t klaunch[FREDOPT_KCLASS_N] = {0};
  int64_t launches = 0;  // kernels enqueued (graph replays count their nodes)
};

namespace {

const char* kErrNames[] = {"ok",        "invalid argument", "shape",     "pattern",
                           "nonfinite", "not loaded",       "out of memory", "cuda error",
                           "timeout",   "unsupported"};

int fail(fredopt_t h, int code, const std::string& msg) {
  if (h) h->last_error = msg;
  return code;
}

int cuda_fail(fredopt_t h, cudaError_t e, const char* what) {
  const int code = (e == cudaErrorMemoryAllocation) ? FREDOPT_ERR_OOM : FREDOPT_ERR_CUDA;
  cudaGetLastError();  // clear non-sticky errors so the handle stays usable
  return fail(h, code, std::string(what) + ": " + cudaGetErrorString(e));
}

#define CK(call)                                       \
  do {                                                 \
    cudaError_t e_ = (call);                           \
    if (e_ != cudaSuccess) return cuda_fail(h, e_, #call); \
  } while (0)

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    cudaGetDevice(&prev);
    if (prev != dev) cudaSetDevice(dev);
  }
  ~DeviceGuard() {
    int cur = -1;
    cudaGetDevice(&cur);
    if (prev >= 0 && cur != prev) cudaSetDevice(prev);
  }
};

bool dev_ptr(uint32_t flags) { return (flags & FREDOPT_DEVICE_PTR) != 0; }

// Order the handle's own stream after the legacy default stream, so device
// inputs written there by the caller are visible.
void join_in(fredopt_t h) {
  if (!h->own_stream) return;
  cudaEventRecord(h->ev_join, 0);
  cudaStreamWaitEvent(h->stream, h->ev_join, 0);
}

cudaError_t copy_in(fredopt_t h, void* dst, const void* src, size_t bytes, uint32_t flags) {
  if (bytes == 0) return cudaSuccess;
  return cudaMemcpyAsync(dst, src, bytes, dev_ptr(flags) ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice,
                         h->stream);
}
cudaError_t copy_out(fredopt_t h, void* dst, const void* src, size_t bytes, uint32_t flags) {
  if (bytes == 0 || !dst) return cudaSuccess;
  return cudaMemcpyAsync(dst, src, bytes, dev_ptr(flags) ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost,
                         h->stream);
}

constexpr size_t kPinStage = 64, kPinBytes = 64 + 64 * 1024;  // error word | staging
constexpr int kStageDoubles = (int)((kPinBytes - kPinStage) / sizeof(double));
double* stage(fredopt_t h) { return reinterpret_cast<double*>(h->pin + kPinStage); }
volatile int* err_word(fredopt_t h) { return reinterpret_cast<volatile int*>(h->pin); }

template <typename T>
cudaError_t upload_vec(fredopt_t h, DBuf<T>& d, const std::vector<T>& v) {
  cudaError_t e = d.alloc(v.size());
  if (e != cudaSuccess) return e;
  if (v.empty()) return cudaSuccess;
  return cudaMemcpyAsync(d.p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice, h->stream);
}

int value_bytes(int fmt) { return fmt == FREDOPT_FP32 ? 4 : 2; }

void free_graph(fredopt_t h) {
  if (h->gexec) cudaGraphExecDestroy(h->gexec);
  if (h->graph) cudaGraphDestroy(h->graph);
  h->gexec = nullptr;
  h->graph = nullptr;
  h->graph_nodes = 0;
  h->graph_timed = false;
  h->gtimers.clear();
}

// ---- timed launch helper ----
Timer& next_timer(fredopt_t h, int cls) {
  if (h->timers_used == h->timers.size()) {
    Timer t;
    cudaEventCreate(&t.a);
    cudaEventCreate(&t.b);
    h->timers.push_back(t);
  }
  Timer& t = h->timers[h->timers_used++];
  t.cls = cls;
  return t;
}

template <class F>
void run(fredopt_t h, int cls, F&& f) {
  if (h->timing) {
    Timer& t = next_timer(h, cls);
    // under stream capture the external flag makes each record a graph node;
    // every replay points those nodes at fresh events (fredopt_iterate)
    const unsigned fl = h->capturing ? cudaEventRecordExternal : cudaEventRecordDefault;
    cudaEventRecordWithFlags(t.a, h->stream, fl);
    f();
    cudaEventRecordWithFlags(t.b, h->stream, fl);
  } else {
    f();
  }
  h->launches += 1;
}

void collect_timers(fredopt_t h) {
  if (!h->timers_used) return;
  cudaStreamSynchronize(h->stream);
  for (size_t i = 0; i < h->timers_used; ++i) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, h->timers[i].a, h->timers[i].b) == cudaSuccess) {
      h->kms[h->timers[i].cls] += ms;
      h->klaunch[h->timers[i].cls] += 1;
    }
  }
  h->timers_used = 0;
}

// Claimed tiles pay off when a pass is long enough for the SMs' different
// streaming rates to matter; in shorter passes the claims cost more than they
// balance (tile_balance 2 claims always).  The lines lie, in nonzeros per
// forward warp, where static and claimed tiles took the same time; per launch,
// static -> claimed, in us:
//   per warp           1.6e4          2.5e4          3.8e4          6.7e4          1.5e5
//   forward FP32       132 -> 133     196 -> 193     293 -> 284     499 -> 473     1071 -> 1026
//   forward 16-bit      85 ->  93     123 -> 130     184 -> 184     306 -> 298      692 ->  640
//   transposed FP32    112 -> 120     170 -> 174     251 -> 251     423 -> 412      890 ->  847
//   transposed 16-bit   89 -> 100     139 -> 146     201 -> 204     339 -> 330      698 ->  662
int64_t claim_min_nnz(fredopt_t h, bool transposed) {
  if (h->fmt == FREDOPT_FP32) return transposed ? 38000 : 20000;
  return transposed ? 48000 : 38000;
}
bool claim_tiles(fredopt_t h, bool transposed) {
  if (h->prm.tile_balance == 2) return true;
  return h->prm.tile_balance == 1 && h->nnz_hot >= claim_min_nnz(h, transposed) * (int64_t)h->geo.fwd_warps;
}

// Passes over every row (whole-GPU shapes).  The double-float final pass does
// about twice the work per nonzero, so claims pay from shorter passes on:
// 7.3e8 nonzeros FP32 1.79 -> 1.41 ms, BF16 1.66 -> 1.18; 7.7e7 (1.6e4 per warp)
// 0.205 -> 0.175; 2.2e7 (4.5e3 per warp) 78.6 -> 77.7 us.  The FP32 product:
// 7.3e8 1.11 -> 1.05 ms, BF16 0.79 -> 0.65; at 7.7e7 equal and BF16 88 -> 94 us.
constexpr int64_t kClaimMinNnzPerWarpFinal = 4096;
bool claim_all_tiles(fredopt_t h, bool final_pass) {
  if (h->prm.tile_balance == 2) return true;
  return h->prm.tile_balance == 1 &&
         h->nnz >= (final_pass ? kClaimMinNnzPerWarpFinal : claim_min_nnz(h, false)) * (int64_t)h->geo_full.fwd_warps;
}

// The kernels of a captured iteration form a dependent chain, each starting
// while its predecessor drains (tiny plan: 62.3 -> 59.9 us per iteration).  Not
// in long passes: CTAs placed early on the SMs that drain first unbalance them
// (1.2e4 nonzeros per warp: 1% slower).  Not for plans that share the GPU, which
// it does not help (six small plans in a batch: 8.42 and 8.40 ms).  Not for single
// calls: a dependent launch costs the host 1 us more (feasibility step of the tiny
// plan: 62.9 against 65.1 us; a gradient of 1.1e7 nonzeros would gain, 83 -> 74 us).
constexpr int64_t kChainMaxNnzPerWarp = 4096;
bool chained(fredopt_t h) {
  return h->capturing && h->nnz_hot < kChainMaxNnzPerWarp * (int64_t)h->geo.fwd_warps &&
         h->geo.n_sms == h->geo_full.n_sms;
}

// number of forward partials
int n_parts(const Geometry& g, const FwdArgs& a) { return a.sched ? a.n_warps : forward_grid(g, a.n_warps); }

// Elements that every array of the CSR, or of the CSC with 16- or 32-bit rows,
// holds (kept buffers differ in length).
int64_t csr_elems(fredopt_t h) {
  const size_t vb = (size_t)value_bytes(h->fmt);
  return (int64_t)std::min({h->col16.p ? h->col16.n : h->col.n, h->Dv.n / vb, h->Lv.n / vb});
}
int64_t csc_elems(fredopt_t h, bool row16) {
  const size_t vb = (size_t)value_bytes(h->fmt);
  return (int64_t)std::min({row16 ? h->crow16.n : h->crow.n, h->DTv.n / vb, h->LTv.n / vb});
}

FwdArgs fwd_args(fredopt_t h, bool hot, bool final_pass = false) {
  FwdArgs a{};
  a.pdl = chained(h);
  a.rp = h->rp.p;
  a.col = h->col.p;
  a.col16 = h->col16.p;
  a.n_elems = csr_elems(h);
  a.Dv = h->Dv.p;
  a.Lv = h->Lv.p;
  a.sD = h->fmt ? h->sD.p : nullptr;
  a.sL = h->fmt ? h->sL.p : nullptr;
  a.warp_row = hot ? h->warp_row_hot.p : h->warp_row_all.p;
  if (hot && claim_tiles(h, false) && h->n_tiles_hot > 0) {
    a.warp_row = h->tile_row_hot.p;
    a.sched = h->fsched.p;
  } else if (!hot && claim_all_tiles(h, final_pass)) {
    a.warp_row = h->tile_row_all.p;
    a.sched = h->fsched.p;
  }
  a.n_x = h->n;
  a.n_x_pad = h->n_pad;
  a.mask = h->mask.p;
  a.n_hot = h->n_hot;
  a.n_warps = a.sched ? (hot ? h->n_tiles_hot : h->n_tiles_all) : hot ? h->geo.fwd_warps : h->geo_full.fwd_warps;
  a.part_stride = n_parts(h->geo, a);
  a.st = h->st.p;
  a.voxel = h->perm ? h->voxel.p : nullptr;
  return a;
}

BwdArgs bwd_args(fredopt_t h, const float2* coef) {
  BwdArgs b{};
  b.st = h->st.p;
  b.n_rows = h->n_hot;
  b.n_elems = csc_elems(h, h->crow16.p != nullptr);
  b.n_ovf = (int32_t)h->n_wide_blocks;
  b.row = h->crow.p;
  b.row16 = h->crow16.p;
  b.hdr = h->chdr.p;
  b.ovf = h->covf.p;
  b.Dv = h->DTv.p;
  b.Lv = h->LTv.p;
  b.chunk_ptr = h->chunk_ptr.p;
  b.warp_chunk = h->warp_chunk.p;
  b.coef = coef;
  b.chunk_sum = h->chunk_sum.p;
  b.n_warps = h->geo.bwd_warps;
  b.pdl = chained(h);
  if (claim_tiles(h, true) && h->n_tiles_bwd > 0) {
    b.warp_chunk = h->tile_chunk.p;
    b.n_warps = h->n_tiles_bwd;
    b.sched = h->bsched.p;
  }
  return b;
}

ColArgs col_args(fredopt_t h) {
  ColArgs c{};
  c.col_chunk = h->col_chunk.p;
  c.chunk_sum = h->chunk_sum.p;
  c.n = h->n;
  c.k2part = h->part.p + h->off_k2;
  c.k2_blocks = con_grid(h->geo, h->n_con_rows);
  c.pdl = chained(h);
  c.W_all = h->W_all;
  c.st = h->st.p;
  c.log = h->log.p;
  c.use_u = 1;
  return c;
}

ConArgs con_args(fredopt_t h) {
  ConArgs c{};
  c.yw = h->yw.p;
  c.mask = h->mask.p;
  c.dd = h->mdd.p;
  c.ll = h->mll.p;
  c.dl = h->mdl.p;
  c.sD = h->fmt ? h->sD.p : nullptr;
  c.sL = h->fmt ? h->sL.p : nullptr;
  c.pdl = chained(h);
  c.rows = h->con_rows.p;
  c.n_list = h->n_con_rows;
  c.gam = h->gam.p;
  c.part = h->part.p + h->off_k2;
  c.st = h->st.p;
  return c;
}


// 1 / priority sum of the sweep blocks' reachable rows.  Formed when the blocks
// are built, and again when the constraint table or c_cdl changes.
void sweep_weights(fredopt_t h) {
  launch_sweep_weights(h->tab, h->con_rows.p, h->n_con_ne, h->sw->size, h->sw->nb, h->mask.p, h->mdd.p, h->mll.p,
                       h->mdl.p, h->sw->wpart.p, h->sw->w.p, h->stream);
}

// Whether the streaming forward product takes the rows of a sweep's nb blocks, with
// the rows between them.  k_sweep_rows takes the structure rows alone, a few entries
// per lane in flight, and a warp at least per row; the other keeps more in flight,
// but stages all of x per block, leaves its successor no room to start early, and
// streams a row with one warp.  Estimates in us per block, fitted to the times of
// whole sweeps, k_sweep_rows / streaming:
//   5.7e7 nonzeros, 23 thousand rows, FP32    1 block 285 / 277    2 318 / 330    3 338 / 356
//   8.0e7, 79 thousand rows                   FP32: 1 374 / 347, 4 493 / 487, 8 570 / 607;  BF16: 350 / 284, 474 / 423, 547 / 544
//   2.6e7, 2.8e6 rows, FP32                   1 1894 / 1298    16 2022 / 1448    32 2116 / 1988    100 2789 / 5314
//   7.5e7, 3765 rows, FP32                    1 373 / 358    2 457 / 465    4 607 / 725
//   4.2e7 of 7.7e7 in structure rows, FP32    1 283 / 320
bool sweep_streams(fredopt_t h, int nb) {
  const bool fp32 = h->fmt == FREDOPT_FP32;
  const double rows = ((double)h->con_nnz / 5.4e5 + (double)h->n_con_ne * 0.28e-3) / nb;
  const double all = ((double)h->nnz_hot + 64.0 * (double)h->n_hot_ne) / (fp32 ? 7.0e5 : 1.2e6) / nb;
  const double row = (double)h->con_nnz / (double)h->n_con_ne / (fp32 ? 250.0 : 400.0);
  return 15.0 + std::max(all, row) < rows;
}

// Blocks of the block-iterative sweep: the streamed rows with nonzeros that
// lie in some structure, in device (= ascending voxel) order, cut into groups
// of S = ceil(count / m) rows.  Builds the CSC position table of the blocks'
// boundaries (the device rows from a block's first structure row to the next
// block's first).
int build_sweep(fredopt_t h, int m) {
  if (h->sw->m == m) return FREDOPT_OK;
  cudaStream_t s = h->stream;
  std::vector<int64_t> C(h->n_con_ne);  // structure rows with nonzeros, ascending
  if (!C.empty()) {
    CK(cudaMemcpyAsync(C.data(), h->con_rows.p, C.size() * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
  }
  std::vector<int64_t> bnd;
  h->sw->m = 0;
  h->sw->nb = 0;
  h->sw->size = 0;
  if (!C.empty()) {
    const int64_t S = ((int64_t)C.size() + m - 1) / m;
    const int nb = (int)(((int64_t)C.size() + S - 1) / S);
    for (int t = 0; t < nb; ++t) bnd.push_back(C[(size_t)t * S]);
    h->sw->nb = nb;
    h->sw->size = S;
  }
  bnd.push_back(C.empty() ? 0 : C.back() + 1);
  h->sw->warps = 0;
  if (!C.empty() && sweep_streams(h, h->sw->nb)) {
    const int W = h->geo_full.fwd_warps;
    CK(h->sw->tiles.alloc(2 * (size_t)W * h->sw->nb));
    for (int t = 0; t < h->sw->nb; ++t)
      launch_tiles(TileArgs{TileArgs::PAIRS, h->rp.p, bnd[t], bnd[t + 1], 0, 0, W, 0, h->row_cost,
                            h->sw->tiles.p + 2 * (size_t)W * t, nullptr}, s);
    h->sw->warps = W;
  }
  CK(upload_vec(h, h->sw->bounds, bnd));
  CK(h->sw->pos.alloc(bnd.size() * h->n));
  if (h->sw->nb > 0)
    launch_sweep_pos(h->cp.p, h->crow.p, h->n, h->sw->bounds.p, (int)bnd.size(), h->sw->pos.p, s);
  CK(h->sw->w.alloc(h->sw->nb));
  CK(h->sw->wpart.alloc((size_t)h->sw->nb * sweep_weight_slices(h->sw->size)));
  CK(h->sw->part.alloc((size_t)((h->sw->size + kSweepConThreads - 1) / kSweepConThreads)));
  CK(h->xs.ensure(h->n_pad));
  CK(cudaMemsetAsync(h->xs.p, 0, h->n_pad * sizeof(float), s));
  CK(h->ys.ensure(h->n_hot));
  sweep_weights(h);
  h->sw->own_entries = 0.0;
  if (h->sw->nb > 0) {
    CK(h->sw->lens.alloc(2 * (size_t)h->sw->nb));
    launch_sweep_lengths(h->sw->pos.p, h->n, h->sw->nb, h->sw->lens.p, s);
    std::vector<double> len(2 * (size_t)h->sw->nb);
    CK(cudaMemcpyAsync(len.data(), h->sw->lens.p, len.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    double s1 = 0.0, s2 = 0.0;
    for (int t = 0; t < h->sw->nb; ++t) {
      s1 += len[2 * t];
      s2 += len[2 * t + 1];
    }
    h->sw->own_entries = s1 > 0.0 ? s2 / s1 : 0.0;
  }
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(s));
  h->sw->m = m;
  return FREDOPT_OK;
}

// One block-iterative sweep from x = w + coef * g (use_coef) or x = w, into out.
void enqueue_sweep(fredopt_t h, const float* w, int use_coef, double lam, double prio_scale, int norm,
                   int in_solve, float* out) {
  cudaStream_t s = h->stream;
  run(h, 5, [&] { launch_sweep_start(h->n, w, h->g.p, use_coef, h->xs.p, h->st.p, s); });
  SweepArgs a{};
  a.list = h->con_rows.p;
  a.n_rows = h->n_hot;
  a.n_elems = csr_elems(h);
  a.n_csc = csc_elems(h, false);
  a.rp = h->rp.p;
  a.col = h->col.p;
  a.col16 = h->col16.p;
  a.rD = h->Dv.p;
  a.rL = h->Lv.p;
  a.sD = h->fmt ? h->sD.p : nullptr;
  a.sL = h->fmt ? h->sL.p : nullptr;
  a.mask = h->mask.p;
  a.dd = h->mdd.p;
  a.ll = h->mll.p;
  a.dl = h->mdl.p;
  a.y = h->ys.p;
  a.gam = h->gam.p;
  a.part = h->sw->part.p;
  a.row = h->crow.p;
  a.Dv = h->DTv.p;
  a.Lv = h->LTv.p;
  a.x = h->xs.p;
  a.n = h->n;
  a.norm = norm;
  a.lam = lam;
  a.prio_scale = prio_scale;
  a.in_solve = in_solve;
  a.st = h->st.p;
  const double row_nnz = h->n_con_ne > 0 ? (double)h->con_nnz / (double)h->n_con_ne : 0.0;
  const double col_nnz = (double)h->nnz_hot / ((double)std::max(1, h->sw->nb) * (double)h->n);
  for (int t = 0; t < h->sw->nb; ++t) {
    a.i0 = t * h->sw->size;
    a.i1 = std::min(h->n_con_ne, a.i0 + h->sw->size);
    a.con_blocks = (int)((a.i1 - a.i0 + kSweepConThreads - 1) / kSweepConThreads);
    a.winv = h->sw->w.p + t;
    a.pos0 = h->sw->pos.p + (size_t)t * h->n;
    a.pos1 = h->sw->pos.p + (size_t)(t + 1) * h->n;
    if (h->sw->warps > 0) {
      FwdArgs fa = fwd_args(h, true);
      fa.pdl = true;
      fa.warp_row = h->sw->tiles.p + 2 * (size_t)h->sw->warps * t;
      fa.n_warps = h->sw->warps;
      fa.sched = nullptr;
      fa.x = h->xs.p;
      fa.y = h->ys.p;
      run(h, 0, [&] { launch_forward(h->geo_full, h->fmt, EPI_STORE, h->hint_fwd, fa, h->tab, s); });
    } else {
      run(h, 0, [&] { launch_sweep_rows(h->fmt, row_nnz, a, s); });
    }
    run(h, 2, [&] { launch_sweep_con(h->tab, a, s); });
    run(h, 1, [&] { launch_sweep_cols(h->fmt, col_nnz, h->sw->own_entries, a, s); });
  }
  run(h, 3, [&] { launch_sweep_finish(h->geo, h->n, h->xs.p, out, in_solve, h->st.p, h->log.p, s); });
}

// One superiorized iteration (Fig. 3 around the simultaneous Fig. 2).
void enqueue_iteration(fredopt_t h) {
  const Geometry& G = h->geo;
  const Tables& t = h->tab;
  cudaStream_t s = h->stream;
  const int N = h->prm.reductions;
  const bool pert = N > 0 && t.n_obj > 0;
  double* part_f = h->part.p + h->off_f;
  double* part_bc = h->part.p + h->off_bc;
  double* part_g = h->part.p + h->off_g;
  FwdArgs fa = fwd_args(h, true);
  fa.x = h->w.p;
  fa.y = h->yw.p;
  if (pert) {
    fa.r_out = h->r.p;
    fa.part = part_f;
    run(h, 0, [&] { launch_forward(G, h->fmt, EPI_OBJ, h->hint_fwd, fa, t, s); });
    for (int step = 0; step < N; ++step) {
      int nf = n_parts(G, fa);
      if (step > 0) {
        run(h, 5, [&] { launch_apply_step(h->n_hot, h->n, h->w.p, h->g.p, h->yw.p, h->yg.p, h->st.p, s); });
        run(h, 5, [&] {
          launch_row_objective(G, t, h->yw.p, h->mask.p, fa.sD, fa.sL, h->n_hot, h->r.p, part_f, s);
        });
        nf = G.row_blocks;
      }
      BwdArgs ba = bwd_args(h, h->r.p);
      run(h, 1, [&] { launch_backward(G, h->fmt, h->hint_bwd, h->obj_dose, ba, s); });
      ColArgs ca = col_args(h);
      ca.out = h->g.p;
      ca.part = part_g;
      run(h, 3, [&] { launch_colfinish(G, COL_GRAD, ca, s); });
      FwdArgs fb = fa;
      fb.x = h->g.p;
      fb.y = h->yg.p;
      fb.r_in = h->r.p;
      fb.r_out = nullptr;
      fb.part = part_bc;
      run(h, 0, [&] { launch_forward(G, h->fmt, EPI_BC, h->hint_fwd, fb, t, s); });
      run(h, 4, [&] {
        launch_finish(step, part_f, nf, part_bc, n_parts(G, fa), part_g, col_grid(G, h->n), h->st.p,
                      h->part.p + h->off_stage, h->part.p + h->off_btab, kBetaTable, chained(h), s);
      });
    }
  } else {
    run(h, 0, [&] { launch_forward(G, h->fmt, EPI_STORE, h->hint_fwd, fa, t, s); });
  }
  if (h->prm.sweep_blocks > 0 && t.n_con > 0) {
    enqueue_sweep(h, h->w.p, pert ? 1 : 0, h->lam, 1.0, h->prm.cimmino_norm, 1, h->w.p);
    return;
  }
  ConArgs k2 = con_args(h);
  k2.yg = pert ? h->yg.p : nullptr;
  k2.use_coef = pert ? 1 : 0;
  run(h, 2, [&] { launch_constraints(G, t, k2, s); });
  if (t.n_con > 0) {
    BwdArgs bb = bwd_args(h, h->gam.p);
    run(h, 1, [&] { launch_backward(G, h->fmt, h->hint_bwd, true, bb, s); });
  }
  ColArgs cc = col_args(h);
  cc.w = h->w.p;
  cc.w_out = h->w.p;
  cc.g = h->g.p;
  cc.use_coef = pert ? 1 : 0;
  cc.use_u = t.n_con > 0 ? 1 : 0;
  cc.norm = h->prm.cimmino_norm;
  cc.lam = h->lam;
  cc.in_solve = 1;
  // norm ALL without decay: the scale lam eta^k / W_all is fixed (the same
  // FP64 operations the kernel would do)
  cc.has_scale = (cc.norm != FREDOPT_NORM_VIOLATED && h->prm.eta == 1.0) ? 1 : 0;
  cc.scale = h->W_all > 0.0 ? cc.lam * 1.0 / h->W_all : 0.0;
  cc.log_block = cc.has_scale;
  run(h, 3, [&] { launch_colfinish(G, COL_PROJ, cc, s); });
}

// Tile weights: a row end or a chunk end (warp reductions and bookkeeping) costs
// about as much as streaming this many nonzeros; 16-bit values stream faster.
// fredopt_autotune picks among the candidates, which hold the weights of a load.
// Measured over the clinical, tiny, half-resolution and batched plans: 128 against
// 64 for 16-bit rows, six plans 8.57 -> 8.38 ms; 64 against 16 per chunk, clinical
// plan in ROI rows 20.75 -> 20.69 ms, an ROI plan of 1e7 nonzeros 2.46 -> 2.40.
constexpr int64_t kRowCosts[] = {16, 32, 64, 128, 256, 512}, kChunkCosts[] = {4, 16, 64, 256, 1024};
constexpr int64_t kRowCost = 64, kRowCost16 = 128, kChunkCost = 64;
template <size_t N>
constexpr bool among(const int64_t (&list)[N], int64_t v) {
  for (int64_t x : list)
    if (x == v) return true;
  return false;
}
static_assert(among(kRowCosts, kRowCost) && among(kRowCosts, kRowCost16) && among(kChunkCosts, kChunkCost),
              "fredopt_autotune can keep the weights of a load");

// Warp partitions.  A segment's sum does not depend on which warp streams it
// (lanes take elements by their absolute block-aligned position and add them
// in order), so these weights change the speed, never a result bit.
int set_fwd_schedule(fredopt_t h, int64_t row_cost) {
  const int W = h->geo.fwd_warps;
  const int64_t *rp = h->rp.p, hot = h->n_hot_ne, cold = h->n_cold_ne;
  CK(h->warp_row_hot.fit(2 * (size_t)W));
  // every row: single products and final passes use the whole GPU whatever
  // the plan's launch shapes (a row's sums do not depend on them)
  const int A = h->geo_full.fwd_warps;
  CK(h->warp_row_all.fit(2 * (size_t)A));
  CK(h->tile_row_hot.fit(2 * (size_t)kGuidedTilesPerWarp * W));
  launch_tiles(TileArgs{TileArgs::PAIRS, rp, 0, hot, 0, 0, W, 0, row_cost, h->warp_row_hot.p, nullptr}, h->stream);
  // the warps shared between streamed and other rows by their cost
  const double c0 = (double)h->nnz_hot + (double)row_cost * (double)hot;
  const double c1 = (double)(h->nnz - h->nnz_hot) + (double)row_cost * (double)cold;
  int w0 = hot > 0 || cold == 0 ? A : 0;
  if (hot > 0 && cold > 0) w0 = std::max(1, std::min(A - 1, (int)std::llround(A * (c0 / (c0 + c1)))));
  launch_tiles(TileArgs{TileArgs::PAIRS, rp, 0, hot, h->n_hot, h->n_hot + cold, w0, A - w0, row_cost,
                        h->warp_row_all.p, nullptr}, h->stream);
  launch_tiles(TileArgs{TileArgs::GUIDED_PAIRS, rp, 0, hot, 0, 0, W, 0, row_cost, h->tile_row_hot.p, nullptr},
               h->stream);
  CK(h->tile_row_all.fit(2 * (size_t)kGuidedTilesPerWarp * A));
  if (w0 > 0)
    launch_tiles(TileArgs{TileArgs::GUIDED_PAIRS, rp, 0, hot, 0, 0, w0, 0, row_cost, h->tile_row_all.p, nullptr},
                 h->stream);
  if (w0 < A)
    launch_tiles(TileArgs{TileArgs::GUIDED_PAIRS, rp, h->n_hot, h->n_hot + cold, 0, 0, A - w0, 0, row_cost,
                          h->tile_row_all.p + 2 * (size_t)kGuidedTilesPerWarp * w0, nullptr}, h->stream);
  h->n_tiles_all = kGuidedTilesPerWarp * A;
  CK(cudaGetLastError());
  h->n_tiles_hot = kGuidedTilesPerWarp * W;
  h->row_cost = row_cost;
  return FREDOPT_OK;
}

int set_bwd_schedule(fredopt_t h, int64_t chunk_cost) {
  const int W = h->geo.bwd_warps;
  const int64_t* cp = h->chunk_ptr.p;
  CK(h->warp_chunk.fit((size_t)W + 1));
  CK(h->tile_chunk.fit((size_t)kGuidedTilesPerWarp * W + 1));
  launch_tiles(TileArgs{TileArgs::BOUNDS32, cp, 0, h->n_chunks, 0, 0, W, 0, chunk_cost, nullptr, h->warp_chunk.p},
               h->stream);
  // claimed tiles: guided sizes over the chunks (the same rule as the forward rows)
  launch_tiles(TileArgs{TileArgs::GUIDED32, cp, 0, h->n_chunks, 0, 0, W, 0, chunk_cost, nullptr, h->tile_chunk.p},
               h->stream);
  CK(cudaGetLastError());
  h->n_tiles_bwd = kGuidedTilesPerWarp * W;
  h->chunk_cost = chunk_cost;
  return FREDOPT_OK;
}

// Objective (Eq. 2 terms) of the streamed rows without nonzeros: their dose
// and LET-weighted dose are 0 for every w, so each term contributes w*T^2 per
// such row of its structure.
double f_empty(fredopt_t h) {
  double f = 0.0;
  for (int i = 0; i < h->tab.n_obj; ++i)
    f += h->tab.obj[i].weight * h->tab.obj[i].target * h->tab.obj[i].target * (double)h->empty_bits[h->tab.obj[i].bit];
  return f;
}

int need_loaded(fredopt_t h) {
  if (!h) return FREDOPT_ERR_INVALID_ARG;
  if (!h->loaded) return fail(h, FREDOPT_ERR_NOT_LOADED, "no influence matrices loaded");
  return FREDOPT_OK;
}

// A spot vector as the forward product takes it: the caller's device array in
// place when the bulk copy of x can read it (16-byte aligned, no padding), else
// a copy in xbuf.
int spot_in(fredopt_t h, const float* src, uint32_t flags, const float** x) {
  *x = src;
  if (dev_ptr(flags) && h->n == h->n_pad && (reinterpret_cast<uintptr_t>(src) & 15) == 0) return FREDOPT_OK;
  CK(copy_in(h, h->xbuf.p, src, (size_t)h->n * sizeof(float), flags));
  *x = h->xbuf.p;
  return FREDOPT_OK;
}

// Sum of squares of n values in the order of k_check_spots: 256 interleaved sums
// (exact products), each 32 joined by halves, then the eight in order.
double slice_squares(const float* x, int32_t n) {
  double v[256] = {0.0};
  for (int32_t j = 0; j < n; ++j) v[j & 255] += (double)x[j] * (double)x[j];
  double sum = 0.0;
  for (int w = 0; w < 8; ++w) {
    double* t = v + 32 * w;
    for (int o = 16; o > 0; o >>= 1)
      for (int l = 0; l < o; ++l) t[l] += t[l + o];
    sum = w ? sum + t[0] : t[0];
  }
  return sum;
}

// Checks w0 (host or device) and sums its squares into *nrm; a host and a device
// array give the same bits and the same error, that of the first bad element.
int check_spots(fredopt_t h, const float* w0, uint32_t flags, double* nrm) {
  double part[2 * kSpotSlices];
  if (dev_ptr(flags)) {
    double* pw = h->part.p + h->off_fin;
    launch_check_spots(w0, h->n, pw, h->stream);
    CK(cudaGetLastError());
    CK(cudaMemcpyAsync(stage(h), pw, sizeof(part), cudaMemcpyDeviceToHost, h->stream));
    CK(cudaStreamSynchronize(h->stream));
    std::memcpy(part, stage(h), sizeof(part));
  } else {
    const int32_t per = (h->n + kSpotSlices - 1) / kSpotSlices;
    for (int b = 0; b < kSpotSlices; ++b) {
      const int64_t j0 = std::min<int64_t>(h->n, (int64_t)b * per), j1 = std::min<int64_t>(h->n, j0 + per);
      part[2 * b] = slice_squares(w0 + j0, (int32_t)(j1 - j0));
      part[2 * b + 1] = (double)kNoSpot;
      bool bad = false;
      for (int64_t j = j0; j < j1; ++j) bad |= !(w0[j] >= 0.0f && w0[j] <= std::numeric_limits<float>::max());
      for (int64_t j = j0; bad && j < j1; ++j) {
        const bool neg = w0[j] < 0.0f && std::isfinite(w0[j]);
        if (!neg && std::isfinite(w0[j])) continue;
        part[2 * b + 1] = (double)(2 * j + neg);
        break;
      }
    }
  }
  double first = (double)kNoSpot;
  for (int b = 0; b < kSpotSlices; ++b) {
    *nrm += part[2 * b];
    first = std::min(first, part[2 * b + 1]);
  }
  if (first == (double)kNoSpot) return FREDOPT_OK;
  if ((unsigned long long)first & 1) return fail(h, FREDOPT_ERR_INVALID_ARG, "w0 must be >= 0");
  return fail(h, FREDOPT_ERR_NONFINITE, "w0 not finite");
}

// Where a kernel writes a spot vector for the caller: the caller's device array
// (unless it overlaps `src`, read by the same kernel, in another way than
// exactly), else `buf`, to be copied out.
float* spot_out(fredopt_t h, float* dst, uint32_t flags, DBuf<float>& buf, const float* src = nullptr) {
  if (!dst || !dev_ptr(flags)) return buf.p;
  const uintptr_t d = reinterpret_cast<uintptr_t>(dst), x = reinterpret_cast<uintptr_t>(src);
  const uintptr_t bytes = (uintptr_t)h->n * sizeof(float);
  if (src && d != x && d < x + bytes && x < d + bytes) return buf.p;
  return dst;
}

// The error word, and the tile counters, which a pass that gave up may have left
// set.  Nothing of the handle is in flight.
void clear_error(fredopt_t h) {
  *err_word(h) = 0;
  if (h->fsched.p) cudaMemsetAsync(h->fsched.p, 0, 2 * sizeof(unsigned int), h->stream);
  if (h->bsched.p) cudaMemsetAsync(h->bsched.p, 0, 2 * sizeof(unsigned int), h->stream);
}

int check_sticky(fredopt_t h) {
  cudaError_t e = cudaStreamSynchronize(h->stream);
  if (e != cudaSuccess) return cuda_fail(h, e, "stream synchronize");
  const int err = *err_word(h);
  if (err) {
    clear_error(h);
    if (err & 2) return fail(h, FREDOPT_ERR_PATTERN, "checked build: an index or tile range out of bounds");
    return fail(h, FREDOPT_ERR_TIMEOUT, "a bounded device-side wait gave up (bulk copy)");
  }
  return FREDOPT_OK;
}

// CTAs of the passes over the listed structure rows
int list_blocks(fredopt_t h) {
  return (int)std::max<int64_t>(1, std::min<int64_t>(std::min(608, h->geo_full.row_blocks), (h->n_con_rows + 255) / 256));
}

int ready_y64(fredopt_t h) {
  const size_t n = (size_t)std::max<int64_t>(1, h->V);
  if (!h->y64.p || h->y64.n < n) h->y64_zeroed = false;
  CK(h->y64.ensure(n));
  if (!h->y64_zeroed) CK(cudaMemsetAsync(h->y64.p, 0, n * sizeof(double2), h->stream));
  h->y64_zeroed = true;
  return FREDOPT_OK;
}

// Double-float pass for w (host or device per flags; null = the current
// iterate of a begun solve) into y64, as in fredopt_end: over every row, or for the
// structure rows over those alone (one row per tile, claimed in order) where that
// takes less time.
int final_pass_y64(fredopt_t h, const float* w, uint32_t flags, bool structures) {
  cudaStream_t s = h->stream;
  const float* x = nullptr;
  if (w) {
    const int rc = spot_in(h, w, flags, &x);
    if (rc) return rc;
  } else {
    if (!h->begun) return fail(h, FREDOPT_ERR_NOT_LOADED, "w is null and no solve is begun");
    x = h->w.p;
  }
  const int rc = ready_y64(h);
  if (rc) return rc;
  FwdArgs fa = fwd_args(h, false, true);
  fa.x = x;
  fa.y64 = h->y64.p;
  fa.dose_out = nullptr;
  fa.letd_out = nullptr;
  if (structures && h->n_con_ne == 0) return FREDOPT_OK;  // every structure value is 0
  // (a listed row restarts a warp's load chain: about 2.7 us of its time, in which it
  // streams 300 nonzeros; a row end in a run of rows costs 64.  3e6 rows of 9, all in
  // structures: 1.71 -> 0.43 ms; the clinical plan's 23 thousand rows of 6e6 98 us)
  if (structures && (double)h->con_nnz + 300.0 * (double)h->n_con_ne <
                        (double)h->nnz + 64.0 * (double)(h->n_hot_ne + h->n_cold_ne)) {
    fa.rows = h->con_rows.p;
    fa.sched = h->fsched.p;
    fa.n_warps = (int32_t)h->n_con_ne;
  }
  run(h, 0, [&] { launch_forward(h->geo_full, h->fmt, EPI_FINAL, false, fa, h->tab, s); });
  CK(cudaGetLastError());
  return FREDOPT_OK;
}

float key_to_float(uint32_t key) {
  const uint32_t u = (key & 0x80000000u) ? (key & 0x7fffffffu) : ~key;
  float f;
  std::memcpy(&f, &u, sizeof(f));
  return f;
}

size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

// =================================================================== ABI

extern "C" {

void fredopt_default_params(fredopt_params* p) {
  if (!p) return;
  std::memset(p, 0, sizeof(*p));
  p->beta0 = -1.0;
  p->eta = 1.0;
  p->reductions = 1;
  p->max_trials = 50;
  p->cimmino_norm = FREDOPT_NORM_ALL;
  p->grad_normalize = 1;
  p->c_cdl = 0.04;
  p->log_capacity = 4096;
  p->use_graphs = 1;
  p->tile_balance = 1;
}

const char* fredopt_strerror(int code) {
  const int i = -code;
  if (i < 0 || i >= (int)(sizeof(kErrNames) / sizeof(kErrNames[0]))) return "unknown error";
  return kErrNames[i];
}

const char* fredopt_last_error(fredopt_t h) { return h ? h->last_error.c_str() : "null handle"; }

int fredopt_create(fredopt_t* out, int device, void* cuda_stream) {
  if (!out) return FREDOPT_ERR_INVALID_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return FREDOPT_ERR_INVALID_ARG;
  }
  fredopt_ctx* h = new fredopt_ctx();
  h->device = device;
  DeviceGuard dg(device);
  if (init_kernels(&h->geo_full, device) != 0) {
    delete h;
    cudaGetLastError();
    return FREDOPT_ERR_CUDA;
  }
  h->geo = h->geo_full;
  int l2 = 0;
  cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, device);
  h->l2_bytes = (size_t)l2;
  if (cuda_stream) {
    h->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  } else {
    if (cudaStreamCreateWithFlags(&h->stream, cudaStreamNonBlocking) != cudaSuccess) {
      delete h;
      return FREDOPT_ERR_CUDA;
    }
    h->own_stream = true;
  }
  if (cudaEventCreateWithFlags(&h->ev_join, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreate(&h->ev_it0) != cudaSuccess || cudaEventCreate(&h->ev_it1) != cudaSuccess ||
      h->st.alloc(1) != cudaSuccess || h->errw.alloc(1) != cudaSuccess ||
      cudaHostAlloc(reinterpret_cast<void**>(&h->pin), kPinBytes, cudaHostAllocMapped) != cudaSuccess ||
      cudaHostGetDevicePointer(reinterpret_cast<void**>(&h->err_dev), h->pin, 0) != cudaSuccess) {
    fredopt_destroy(h);
    return FREDOPT_ERR_CUDA;
  }
  *err_word(h) = 0;
  h->st_host.err = h->err_dev;
  cudaMemcpyAsync(h->st.p, &h->st_host, sizeof(DevState), cudaMemcpyHostToDevice, h->stream);
  fredopt_default_params(&h->prm);
  h->tab.c = 0.04;
  cudaStreamSynchronize(h->stream);
  *out = h;
  return FREDOPT_OK;
}

int fredopt_destroy(fredopt_t h) {
  if (!h) return FREDOPT_ERR_INVALID_ARG;
  DeviceGuard dg(h->device);
  if (h->stream) cudaStreamSynchronize(h->stream);
  free_graph(h);
  for (auto& t : h->timers) {
    cudaEventDestroy(t.a);
    cudaEventDestroy(t.b);
  }
  if (h->ev_join) cudaEventDestroy(h->ev_join);
  if (h->ev_it0) cudaEventDestroy(h->ev_it0);
  if (h->ev_it1) cudaEventDestroy(h->ev_it1);
  cudaStream_t own = h->own_stream ? h->stream : nullptr;
  if (h->pin) cudaFreeHost(h->pin);
  delete h;  // frees every device buffer
  if (own) cudaStreamDestroy(own);
  return FREDOPT_OK;
}

// Frees what a plan's size determines.
static void release_plan(fredopt_t h) {
  h->rp.release(); h->col.release(); h->col16.release(); h->Dv.release(); h->Lv.release();
  h->sD.release(); h->sL.release(); h->mdd.release(); h->mll.release(); h->mdl.release();
  h->voxel.release(); h->mask.release(); h->con_rows.release(); h->cp.release(); h->covf.release();
  h->crow.release(); h->crow16.release(); h->chdr.release(); h->DTv.release(); h->LTv.release();
  h->yw.release(); h->yg.release(); h->r.release(); h->gam.release(); h->ucoef.release();
  h->y64.release(); h->yall.release(); h->fout_a.release(); h->fout_b.release();
  h->vin_a.release(); h->vin_b.release(); h->ys.release(); h->sw.reset(new Sweep());
}

static int load_influence(fredopt_t h, int64_t n_vox, int32_t n_spots, int64_t nnz,
                           const int64_t* row_ptr, const int32_t* col, const float* D_val,
                           const float* L_val, const uint32_t* voxel_mask, int format,
                           uint32_t flags, bool* keep) {
  if (!h) return FREDOPT_ERR_INVALID_ARG;
  const int fmt = format & 0xff;
  const bool roi = (format & FREDOPT_ROWS_ROI) != 0;
  if (fmt < 0 || fmt > 2 || (format & ~0x7ff))
    return fail(h, FREDOPT_ERR_INVALID_ARG, "format must be FP32/BF16/FP16 | ROWS_ALL/ROI | INDEX32 | SHARED");
  if (n_vox < 0 || n_spots < 1 || nnz < 0 || nnz > 2147483647LL || n_vox > 2147483647LL)
    return fail(h, FREDOPT_ERR_SHAPE, "need n_vox >= 0, n_spots >= 1, 0 <= nnz < 2^31");
  if (!row_ptr || !voxel_mask || (nnz > 0 && (!col || !D_val || !L_val)))
    return fail(h, FREDOPT_ERR_INVALID_ARG, "null array");
  DeviceGuard dg(h->device);
  free_graph(h);
  h->loaded = false;
  h->begun = false;
  h->sw->m = 0;
  cudaStream_t s = h->stream;
  if (!*keep) release_plan(h);
  join_in(h);
  const bool host = !dev_ptr(flags);
  const int vb = value_bytes(fmt);
  // every index / value array is zero padded past its last nonzero
  const int64_t nnz_alloc = ((nnz + 255) & ~255LL) + kPadElems;

  // ---- row order (and the check of row_ptr), on the device
  DBuf<int64_t> rp_in, row_blk;
  DBuf<uint32_t> mask_in;
  DBuf<RowTotals> tot_rows;
  const int64_t* rpp = row_ptr;
  const uint32_t* mp = voxel_mask;
  if (host) {
    CK(rp_in.alloc(n_vox + 1));
    CK(mask_in.alloc(n_vox));
    CK(cudaMemcpyAsync(rp_in.p, row_ptr, (n_vox + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, s));
    if (n_vox) CK(cudaMemcpyAsync(mask_in.p, voxel_mask, n_vox * sizeof(uint32_t), cudaMemcpyHostToDevice, s));
    rpp = rp_in.p;
    mp = mask_in.p;
  }
  CK(row_blk.alloc(row_order_scratch(n_vox)));
  CK(tot_rows.alloc(1));
  CK(cudaMemsetAsync(tot_rows.p, 0, sizeof(RowTotals), s));
  launch_rows_count(rpp, mp, n_vox, nnz, roi, row_blk.p, tot_rows.p, s);
  CK(cudaGetLastError());
  RowTotals tot;
  CK(cudaMemcpyAsync(&tot, tot_rows.p, sizeof(tot), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (tot.flags & kRowsBadEnds) return fail(h, FREDOPT_ERR_PATTERN, "row_ptr[0] != 0 or row_ptr[n_vox] != nnz");
  if (tot.flags & kRowsNotMonotone) return fail(h, FREDOPT_ERR_PATTERN, "row_ptr not monotone");
  const bool perm = (tot.flags & kRowsPermuted) != 0;
  const int64_t n_hot_ne = tot.c[0], n_hot = tot.c[0] + tot.c[1], n_cold_ne = tot.c[2], nnz_hot = tot.c[3];
  const int64_t nh_alloc = ((nnz_hot + 255) & ~255LL) + kPadElems;

  // ---- the previous plan's buffers: kept where the new plan needs at least
  // half of them (a plan re-planned on the same handle), else all freed first
  const bool similar = *keep && h->Dv.p && h->Dv.n >= (size_t)nnz_alloc * vb && h->Dv.n / 2 <= (size_t)nnz_alloc * vb &&
                       h->DTv.n >= (size_t)nh_alloc * vb && h->DTv.n / 2 <= (size_t)nh_alloc * vb && h->V >= n_vox &&
                       h->V / 2 <= n_vox;
  *keep = similar;
  if (!similar) release_plan(h);
  h->y64_zeroed = h->yall_zeroed = false;
  h->covf.release();
  h->ucoef.release();
  if (fmt == FREDOPT_FP32) {
    h->sD.release();
    h->sL.release();
  }
  h->V = n_vox; h->nnz = nnz; h->n = n_spots; h->n_pad = (n_spots + 3) & ~3;
  h->fmt = fmt; h->roi = roi; h->perm = perm; h->n_hot = n_hot; h->nnz_hot = nnz_hot;
  h->n_hot_ne = n_hot_ne; h->n_cold_ne = n_cold_ne;
  h->n_con_ne = tot.c[5]; h->n_con_rows = tot.c[5] + tot.c[6]; h->con_nnz = (int64_t)tot.con_nnz;
  for (int b = 0; b < 32; ++b) h->empty_bits[b] = tot.empty_bits[b];

  CK(h->rp.fit(n_vox + 1));
  CK(h->mask.fit(n_hot));
  CK(h->con_rows.fit(h->n_con_rows));
  if (perm) CK(h->voxel.fit(n_vox));
  else h->voxel.release();
  if (fmt != FREDOPT_FP32) {
    CK(h->sD.fit(n_vox));
    CK(h->sL.fit(n_vox));
  }
  launch_rows_place(rpp, mp, n_vox, roi, row_blk.p, tot_rows.p, h->rp.p, perm ? h->voxel.p : nullptr, h->mask.p,
                    h->con_rows.p, fmt ? h->sD.p : nullptr, fmt ? h->sL.p : nullptr, s);
  CK(cudaGetLastError());

  // ---- index and value storage.  16-bit column indices for the forward
  // stream (2 bytes less per nonzero, same sums) when x is staged in shared
  // memory (that bounds n_spots below 65536).  FP32 host arrays whose rows
  // keep their order in memory are uploaded into place.
  const bool narrow = !(format & FREDOPT_INDEX32) && n_spots <= 65536 && forward_uses_smem(h->geo_full, h->n_pad);
  if (narrow) {
    h->col.release();
    CK(h->col16.fit(nnz_alloc));
  } else {
    h->col16.release();
    CK(h->col.fit(nnz_alloc));
  }
  CK(h->Dv.fit((size_t)nnz_alloc * vb));
  CK(h->Lv.fit((size_t)nnz_alloc * vb));
  const int ib = narrow ? 2 : 4;
  uint8_t* colp8 = narrow ? reinterpret_cast<uint8_t*>(h->col16.p) : reinterpret_cast<uint8_t*>(h->col.p);
  CK(cudaMemsetAsync(colp8 + nnz * ib, 0, (nnz_alloc - nnz) * ib, s));
  CK(cudaMemsetAsync(h->Dv.p + nnz * vb, 0, (nnz_alloc - nnz) * vb, s));
  CK(cudaMemsetAsync(h->Lv.p + nnz * vb, 0, (nnz_alloc - nnz) * vb, s));
  DBuf<int32_t> col_in;
  DBuf<float> D_in, L_in;
  const int32_t* colp = col;
  const float *Dp = D_val, *Lp = L_val;
  const bool in_place = host && fmt == FREDOPT_FP32 && n_cold_ne == 0;
  if (host) {
    CK(col_in.alloc(nnz));
    float *Dd = reinterpret_cast<float*>(h->Dv.p), *Ld = reinterpret_cast<float*>(h->Lv.p);
    if (!in_place) {
      CK(D_in.alloc(nnz));
      CK(L_in.alloc(nnz));
      Dd = D_in.p;
      Ld = L_in.p;
    }
    if (nnz) {
      CK(cudaMemcpyAsync(col_in.p, col, nnz * sizeof(int32_t), cudaMemcpyHostToDevice, s));
      CK(cudaMemcpyAsync(Dd, D_val, nnz * sizeof(float), cudaMemcpyHostToDevice, s));
      CK(cudaMemcpyAsync(Ld, L_val, nnz * sizeof(float), cudaMemcpyHostToDevice, s));
    }
    colp = col_in.p;
    Dp = Dd;
    Lp = Ld;
  }

  // ---- one pass over the input: validation, storage, FP64-class row moments
  CK(h->mdd.fit(n_hot)); CK(h->mll.fit(n_hot)); CK(h->mdl.fit(n_hot));
  CK(cudaMemsetAsync(h->mdd.p, 0, std::max<int64_t>(1, n_hot) * sizeof(double), s));
  CK(cudaMemsetAsync(h->mll.p, 0, std::max<int64_t>(1, n_hot) * sizeof(double), s));
  CK(cudaMemsetAsync(h->mdl.p, 0, std::max<int64_t>(1, n_hot) * sizeof(double), s));
  CK(cudaMemsetAsync(h->errw.p, 0, sizeof(int), s));
  LoadRowsArgs la{rpp, h->rp.p, perm ? h->voxel.p : nullptr, n_hot, n_hot_ne, n_cold_ne, n_spots, colp, Dp, Lp, colp8,
                  h->Dv.p, h->Lv.p, fmt ? h->sD.p : nullptr, fmt ? h->sL.p : nullptr, h->mdd.p, h->mll.p, h->mdl.p,
                  h->errw.p};
  launch_load_rows(fmt, narrow, !in_place, la, s);
  CK(cudaGetLastError());
  int verr = 0;
  CK(cudaMemcpyAsync(&verr, h->errw.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (verr & 1) return fail(h, FREDOPT_ERR_PATTERN, "column index out of range or not strictly increasing within a row");
  if (verr & 2) return fail(h, FREDOPT_ERR_NONFINITE, "NaN or Inf in D or L");
  col_in.release(); D_in.release(); L_in.release(); rp_in.release(); mask_in.release();

  // ---- launch shapes: the whole GPU, or with FREDOPT_SHARED one SM's
  // worth of CTAs per kSharedNnzPerSm nonzeros, so that the kernels of other
  // plans in a batch or on a server share the GPU (16 plans of 6e5-7e7
  // nonzeros, BF16, one batch graph: 13621 against 10560 plan-iterations/s;
  // 12831, 13205 and 12380 at 1e5, 2e5 and 8e5 nonzeros per SM)
  {
#ifndef FO_SHARED_NNZ_PER_SM
#define FO_SHARED_NNZ_PER_SM 400000
#endif
    constexpr int64_t kSharedNnzPerSm = FO_SHARED_NNZ_PER_SM;
    const Geometry& F = h->geo_full;
    int eff = F.n_sms;
    if (format & FREDOPT_SHARED)
      eff = (int)std::max<int64_t>(1, std::min<int64_t>(F.n_sms, (h->nnz_hot + kSharedNnzPerSm - 1) / kSharedNnzPerSm));
    Geometry g = F;
    g.n_sms = eff;
    g.fwd_blocks = F.fwd_blocks / F.n_sms * eff;
    g.fwd_warps = g.fwd_blocks * (g.fwd_threads / 32);
    g.bwd_blocks = F.bwd_blocks / F.n_sms * eff;
    g.bwd_warps = g.bwd_blocks * (g.bwd_threads / 32);
    g.row_blocks = F.row_blocks / F.n_sms * eff;
    g.col_blocks = F.col_blocks / F.n_sms * eff;
    h->geo = g;
  }

  // ---- CSC copy of the streamed rows (blocked stable counting transpose) and
  // the chunks of the transposed product.  Rows without nonzeros (after the
  // others in device order) add nothing; strips over the whole GPU whatever the
  // plan's launch shapes (the transpose does not depend on its partition).
  {
    const CscShape cs = csc_shape(h->geo_full, fmt, std::max<int64_t>(1, n_hot_ne), n_spots, nnz_hot);
    DBuf<int64_t> strip, tot_d;
    DBuf<int32_t> cnt, split;
    CK(strip.alloc((size_t)cs.n_strip + 1));
    launch_tiles(TileArgs{TileArgs::BOUNDS64, h->rp.p, 0, n_hot_ne, 0, 0, cs.n_strip, 0, 1, strip.p, nullptr}, s);
    CK(cnt.alloc((size_t)cs.n_strip * n_spots));
    CK(cudaMemsetAsync(cnt.p, 0, (size_t)cs.n_strip * n_spots * sizeof(int32_t), s));
    if (cs.use_split) CK(split.alloc((size_t)(cs.n_grp + 1) * cs.n_rows));
    if (n_hot_ne > 0)
      launch_csc_count(cs, h->geo_full.smem_limit, h->rp.p, h->col.p, h->col16.p, strip.p, cnt.p, split.p, s);
    CK(tot_d.alloc(n_spots));
    launch_csc_colsum(cnt.p, cs.n_strip, n_spots, tot_d.p, s);
    int64_t C = nnz_hot / ((int64_t)h->geo.bwd_warps * 8);
    C = std::max<int64_t>(256, std::min<int64_t>(8192, C));
    C = (C + 31) & ~31LL;
    CK(h->cp.fit((size_t)n_spots + 1));
    CK(h->col_chunk.fit((size_t)n_spots + 1));
    launch_csc_columns(tot_d.p, n_spots, C, h->cp.p, h->col_chunk.p, s);
    launch_csc_offsets(cnt.p, cs.n_strip, n_spots, h->cp.p, s);
    const int64_t max_chunks = nnz_hot / C + n_spots;
    CK(h->chunk_ptr.fit((size_t)max_chunks + 1));
    CK(h->chunk_sum.fit((size_t)max_chunks));
    launch_chunk_fill(h->cp.p, h->col_chunk.p, n_spots, C, h->chunk_ptr.p, s);
    CK(h->crow.fit(nh_alloc));
    CK(h->DTv.fit((size_t)nh_alloc * vb));
    CK(h->LTv.fit((size_t)nh_alloc * vb));
    CK(cudaMemsetAsync(h->crow.p + nnz_hot, 0, (nh_alloc - nnz_hot) * sizeof(int32_t), s));
    CK(cudaMemsetAsync(h->DTv.p + (size_t)nnz_hot * vb, 0, (size_t)(nh_alloc - nnz_hot) * vb, s));
    CK(cudaMemsetAsync(h->LTv.p + (size_t)nnz_hot * vb, 0, (size_t)(nh_alloc - nnz_hot) * vb, s));
    int64_t total = 0;
    int32_t n_chunks = 0;
    CK(cudaMemcpyAsync(&total, h->cp.p + n_spots, sizeof(total), cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(&n_chunks, h->col_chunk.p + n_spots, sizeof(n_chunks), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (total != nnz_hot) return fail(h, FREDOPT_ERR_CUDA, "CSC count mismatch");
    h->n_chunks = n_chunks;
    if (n_hot_ne > 0)
      launch_csc_fill(cs, fmt, h->rp.p, h->col.p, h->col16.p, h->Dv.p, h->Lv.p, strip.p, split.p, cnt.p, h->crow.p,
                      h->DTv.p, h->LTv.p, s);
    CK(cudaGetLastError());

    // based 16-bit row indices for the transposed product (2 bytes less per
    // nonzero and pass; crow stays for the sweep and inspection)
    h->n_wide_blocks = 0;
    if (!(format & FREDOPT_INDEX32)) {
      const int64_t n_cblk = nh_alloc / 128;
      CK(h->crow16.fit(nh_alloc));
      CK(h->chdr.fit(n_cblk));
      CK(h->cnw.ensure(2));
      CK(cudaMemsetAsync(h->cnw.p, 0, 2 * sizeof(unsigned int), s));
      launch_narrow_rows(h->crow.p, n_cblk, h->crow16.p, h->chdr.p, h->cnw.p, s);
      CK(cudaGetLastError());
      unsigned int n_wide = 0;
      CK(cudaMemcpyAsync(&n_wide, h->cnw.p, sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
      CK(cudaStreamSynchronize(s));
      CK(h->covf.alloc((size_t)std::max(1u, n_wide) * 128));
      launch_narrow_rows_wide(h->crow.p, n_cblk, h->chdr.p, h->covf.p, h->cnw.p + 1, n_wide, s);
      CK(cudaGetLastError());
      h->n_wide_blocks = n_wide;
    } else {
      h->crow16.release();
    }
    const int rc = set_bwd_schedule(h, kChunkCost);
    if (rc) return rc;
    CK(cudaStreamSynchronize(s));  // the scratch of this block is freed here
  }

  // ---- row schedules of the forward product (rows with nonzeros only)
  CK(h->fsched.ensure(2));
  CK(cudaMemsetAsync(h->fsched.p, 0, 2 * sizeof(unsigned int), s));
  CK(h->bsched.ensure(2));
  CK(cudaMemsetAsync(h->bsched.p, 0, 2 * sizeof(unsigned int), s));
  {
    const int rc = set_fwd_schedule(h, fmt == FREDOPT_FP32 ? kRowCost : kRowCost16);
    if (rc) return rc;
  }
  // streaming (evict-first) loads when the streamed matrices do not fit in L2
  const double mat_bytes = (double)h->nnz_hot * ((h->col16.p ? 2.0 : 4.0) + 2.0 * vb);
#ifndef FO_STREAM_HINT
#define FO_STREAM_HINT -1
#endif
  h->hint_fwd = FO_STREAM_HINT < 0 ? mat_bytes > 0.5 * (double)h->l2_bytes : FO_STREAM_HINT != 0;
  h->hint_bwd = h->hint_fwd;

  // ---- work buffers
  CK(h->w.fit(h->n_pad)); CK(h->g.fit(h->n_pad)); CK(h->xbuf.fit(h->n_pad)); CK(h->gtmp.fit(h->n_pad));
  CK(cudaMemsetAsync(h->w.p, 0, h->n_pad * sizeof(float), s));
  CK(cudaMemsetAsync(h->g.p, 0, h->n_pad * sizeof(float), s));
  CK(cudaMemsetAsync(h->xbuf.p, 0, h->n_pad * sizeof(float), s));
  CK(cudaMemsetAsync(h->gtmp.p, 0, h->n_pad * sizeof(float), s));
  CK(h->yw.fit(n_hot)); CK(h->yg.fit(n_hot)); CK(h->r.fit(n_hot)); CK(h->gam.fit(n_hot));
  // rows without nonzeros are never written by the forward product: keep them 0
  CK(cudaMemsetAsync(h->yw.p, 0, std::max<int64_t>(1, n_hot) * sizeof(float2), s));
  CK(cudaMemsetAsync(h->yg.p, 0, std::max<int64_t>(1, n_hot) * sizeof(float2), s));
  CK(cudaMemsetAsync(h->r.p, 0, std::max<int64_t>(1, n_hot) * sizeof(float2), s));
  // projection coefficients: rows without a structure bit are never written
  CK(cudaMemsetAsync(h->gam.p, 0, std::max<int64_t>(1, n_hot) * sizeof(float2), s));
  const Geometry& G = h->geo;
  // forward partials: one per tile (at most 7 guided tiles per warp)
  const int max_tiles = kGuidedTilesPerWarp * G.fwd_warps;
  h->off_f = 0;
  h->off_bc = h->off_f + std::max(max_tiles, G.row_blocks);
  h->off_g = h->off_bc + 2 * max_tiles;
  h->off_k2 = h->off_g + G.col_blocks;
  h->off_fin = h->off_k2 + 4 * con_grid(G, std::numeric_limits<int64_t>::max() / 2);
  h->off_cnt = h->off_fin + 8 * h->geo_full.row_blocks;
  h->off_stage = h->off_cnt + 3 * h->geo_full.row_blocks;
  h->off_btab = h->off_stage + 4 * kFinishBlocks;
  h->n_part = h->off_btab + kBetaTable;
  h->btab_alpha = -1.0;  // the table is refilled at the next fredopt_begin
  CK(h->part.fit(h->n_part));
  CK(cudaMemsetAsync(h->part.p, 0, h->n_part * sizeof(double), s));
  CK(cudaStreamSynchronize(s));

  h->tab.n_con = 0;
  h->tab.n_obj = 0;
  h->tab.obj_bits = 0u;
  h->have_con = false;
  h->obj_dose = false;
  h->W_all = 0.0;
  h->n_rows_reach = h->n_unreach = 0;
  h->loaded = true;
  return FREDOPT_OK;
}

int fredopt_load_influence(fredopt_t h, int64_t n_vox, int32_t n_spots, int64_t nnz,
                           const int64_t* row_ptr, const int32_t* col, const float* D_val,
                           const float* L_val, const uint32_t* voxel_mask, int format,
                           uint32_t flags) {
  bool keep = true;
  int rc = load_influence(h, n_vox, n_spots, nnz, row_ptr, col, D_val, L_val, voxel_mask, format, flags, &keep);
  if (rc == FREDOPT_ERR_OOM && keep) {  // kept buffers are up to twice what the plan needs: without them
    keep = false;
    rc = load_influence(h, n_vox, n_spots, nnz, row_ptr, col, D_val, L_val, voxel_mask, format, flags, &keep);
  }
  return rc;
}

int fredopt_set_constraints(fredopt_t h, int n, const fredopt_constraint* c) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (n < 0 || n > kMaxCon || (n > 0 && !c)) return fail(h, FREDOPT_ERR_INVALID_ARG, "0 <= n <= 32 constraints");
  for (int i = 0; i < n; ++i) {
    if (c[i].struct_bit >= 32 || c[i].kind < 0 || c[i].kind > 5 || !std::isfinite(c[i].bound) ||
        !(c[i].priority > 0.0) || !std::isfinite(c[i].priority))
      return fail(h, FREDOPT_ERR_INVALID_ARG, "constraint " + std::to_string(i) + " invalid");
  }
  DeviceGuard dg(h->device);
  free_graph(h);
  h->tab.n_con = n;
  for (int i = 0; i < n; ++i) {
    h->tab.con[i].bit = c[i].struct_bit;
    h->tab.con[i].kind = c[i].kind;
    h->tab.con[i].bound = c[i].bound;
    h->tab.con[i].prio = c[i].priority;
  }
  const int fb = list_blocks(h);
  double* pc = h->part.p + h->off_cnt;
  launch_count_rows(fb, h->tab, h->mask.p, h->mdd.p, h->mll.p, h->mdl.p, h->con_rows.p,
                    h->n_con_rows, pc, h->stream);
  CK(cudaGetLastError());
  const double* hp = stage(h);
  CK(cudaMemcpyAsync(stage(h), pc, 3 * fb * sizeof(double), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  double nr = 0, nu = 0, W = 0;
  for (int b = 0; b < fb; ++b) {
    nr += hp[3 * b];
    nu += hp[3 * b + 1];
    W += hp[3 * b + 2];
  }
  h->n_rows_reach = (int64_t)nr;
  h->n_unreach = (int64_t)nu;
  h->W_all = W;
  if (h->sw->m > 0) sweep_weights(h);
  h->have_con = true;
  return FREDOPT_OK;
}

int fredopt_set_objective(fredopt_t h, int n, const fredopt_objective_term* t) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (n < 0 || n > kMaxObj || (n > 0 && !t)) return fail(h, FREDOPT_ERR_INVALID_ARG, "0 <= n <= 32 terms");
  for (int i = 0; i < n; ++i)
    if (t[i].struct_bit >= 32 || (t[i].quantity != FREDOPT_Q_DOSE && t[i].quantity != FREDOPT_Q_CDL) ||
        !std::isfinite(t[i].target) || !(t[i].weight > 0.0) || !std::isfinite(t[i].weight))
      return fail(h, FREDOPT_ERR_INVALID_ARG, "objective term " + std::to_string(i) + " invalid");
  free_graph(h);
  h->tab.n_obj = n;
  h->tab.obj_bits = 0u;
  h->obj_dose = false;
  for (int i = 0; i < n; ++i) {
    h->tab.obj[i].bit = t[i].struct_bit;
    h->tab.obj_bits |= 1u << t[i].struct_bit;
    h->tab.obj[i].q = t[i].quantity;
    h->tab.obj[i].target = t[i].target;
    h->tab.obj[i].weight = t[i].weight;
    if (t[i].quantity == FREDOPT_Q_DOSE) h->obj_dose = true;
  }
  if (h->begun) {
    DeviceGuard dg(h->device);
    h->st_host.f_empty = f_empty(h);
    CK(cudaMemcpyAsync(&h->st.p->f_empty, &h->st_host.f_empty, sizeof(double), cudaMemcpyHostToDevice,
                       h->stream));
    CK(cudaStreamSynchronize(h->stream));
  }
  return FREDOPT_OK;
}

int fredopt_begin(fredopt_t h, const float* w0, double alpha, double relaxation,
                  const fredopt_params* params, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!w0) return fail(h, FREDOPT_ERR_INVALID_ARG, "w0 is null");
  fredopt_params p;
  if (params) p = *params;
  else fredopt_default_params(&p);
  if (!(alpha > 0.0 && alpha < 1.0)) return fail(h, FREDOPT_ERR_INVALID_ARG, "need 0 < alpha < 1");
  if (!(relaxation > 0.0 && relaxation <= 2.0)) return fail(h, FREDOPT_ERR_INVALID_ARG, "need 0 < relaxation <= 2");
  if (!(p.eta > 0.0 && p.eta <= 1.0)) return fail(h, FREDOPT_ERR_INVALID_ARG, "need 0 < eta <= 1");
  if (p.reductions < 0 || p.max_trials < 1 || p.log_capacity < 0 ||
      (p.cimmino_norm != FREDOPT_NORM_ALL && p.cimmino_norm != FREDOPT_NORM_VIOLATED) ||
      !(p.c_cdl > 0.0) || !std::isfinite(p.beta0) || p.sweep_blocks < 0 ||
      p.sweep_blocks > FREDOPT_MAX_SWEEP_BLOCKS || p.tile_balance < 0 || p.tile_balance > 2)
    return fail(h, FREDOPT_ERR_INVALID_ARG, "bad parameters");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  join_in(h);
  double nrm = 0.0;
  if ((rc = check_spots(h, w0, flags, &nrm))) return rc;
  free_graph(h);
  if (p.sweep_blocks > 0) {
    rc = build_sweep(h, p.sweep_blocks);
    if (rc) return rc;
  }
  h->prm = p;
  h->alpha = alpha;
  h->lam = relaxation;
  h->beta0 = p.beta0 < 0.0 ? 0.1 * std::sqrt(nrm) : p.beta0;
  if (h->tab.c != p.c_cdl) {
    h->tab.c = p.c_cdl;
    if (h->sw->m > 0) sweep_weights(h);
  }
  CK(copy_in(h, h->w.p, w0, h->n * sizeof(float), flags));
  if (h->btab_alpha != alpha || h->btab_beta0 != h->beta0) {
    // asynchronous: no allocation or host synchronisation in a served begin
    launch_beta_table(h->part.p + h->off_btab, kBetaTable, h->beta0, alpha, s);
    CK(cudaGetLastError());
    h->btab_alpha = alpha;
    h->btab_beta0 = h->beta0;
  }
  CK(h->log.fit(std::max(1, p.log_capacity)));
  DevState& d = h->st_host;
  std::memset(&d, 0, sizeof(d));
  d.err = h->err_dev;
  d.beta0 = h->beta0;
  d.alpha = alpha;
  d.lam = relaxation;
  d.eta = p.eta;
  d.W_all = h->W_all;
  d.reductions = p.reductions;
  d.max_trials = p.max_trials;
  d.norm = p.cimmino_norm;
  d.grad_normalize = p.grad_normalize ? 1 : 0;
  d.log_cap = p.log_capacity;
  d.f_empty = f_empty(h);
  std::memcpy(stage(h), &d, sizeof(d));
  CK(cudaMemcpyAsync(h->st.p, stage(h), sizeof(DevState), cudaMemcpyHostToDevice, s));
  h->iters_run = 0;
  h->device_ms = 0.0;
  h->it_pending = false;
  if (p.use_graphs) {
    const int64_t before = h->launches;
    const size_t t0 = h->timers_used;
    CK(cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal));
    h->capturing = true;
    enqueue_iteration(h);
    cudaError_t e = cudaStreamEndCapture(s, &h->graph);
    h->capturing = false;
    if (e != cudaSuccess) {
      h->graph = nullptr;
      h->timers_used = t0;
      return cuda_fail(h, e, "graph capture");
    }
    h->graph_nodes = (int)(h->launches - before);
    h->launches = before;
    if (h->timing) {
      // the event-record nodes of the capture, matched to the kernels' timers
      size_t n = 0;
      CK(cudaGraphGetNodes(h->graph, nullptr, &n));
      std::vector<cudaGraphNode_t> nodes(n);
      CK(cudaGraphGetNodes(h->graph, nodes.data(), &n));
      std::vector<std::pair<cudaEvent_t, cudaGraphNode_t>> rec;
      for (cudaGraphNode_t nd : nodes) {
        cudaGraphNodeType ty;
        CK(cudaGraphNodeGetType(nd, &ty));
        if (ty != cudaGraphNodeTypeEventRecord) continue;
        cudaEvent_t ev = nullptr;
        CK(cudaGraphEventRecordNodeGetEvent(nd, &ev));
        rec.emplace_back(ev, nd);
      }
      auto node_of = [&](cudaEvent_t ev) -> cudaGraphNode_t {
        for (auto& r : rec)
          if (r.first == ev) return r.second;
        return nullptr;
      };
      h->gtimers.clear();
      for (size_t i = t0; i < h->timers_used; ++i) {
        GraphTimer g{node_of(h->timers[i].a), node_of(h->timers[i].b), h->timers[i].cls};
        if (!g.a || !g.b) {
          h->timers_used = t0;
          free_graph(h);
          return fail(h, FREDOPT_ERR_CUDA, "timed graph capture: event node missing");
        }
        h->gtimers.push_back(g);
      }
      h->timers_used = t0;  // captured, not recorded: no times to collect
      h->graph_timed = true;
    }
    CK(cudaGraphInstantiate(&h->gexec, h->graph, 0));
  }
  CK(cudaStreamSynchronize(s));
  if (*err_word(h)) clear_error(h);  // of an earlier solve that no call reported
  h->begun = true;
  return FREDOPT_OK;
}

int fredopt_iterate(fredopt_t h, int iters) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!h->begun) return fail(h, FREDOPT_ERR_NOT_LOADED, "call fredopt_begin first");
  if (iters < 0) return fail(h, FREDOPT_ERR_INVALID_ARG, "iters < 0");
  if (iters == 0) return FREDOPT_OK;
  DeviceGuard dg(h->device);
  if (h->it_pending) {
    float ms = 0.f;
    CK(cudaEventSynchronize(h->ev_it1));
    if (cudaEventElapsedTime(&ms, h->ev_it0, h->ev_it1) == cudaSuccess) h->device_ms += ms;
    h->it_pending = false;
  }
  CK(cudaEventRecord(h->ev_it0, h->stream));
  for (int i = 0; i < iters; ++i) {
    if (h->gexec && h->graph_timed == h->timing) {
      // a timed graph records each kernel's events into fresh timers; the
      // update affects this and later launches only
      for (const GraphTimer& g : h->gtimers) {
        Timer& t = next_timer(h, g.cls);
        CK(cudaGraphExecEventRecordNodeSetEvent(h->gexec, g.a, t.a));
        CK(cudaGraphExecEventRecordNodeSetEvent(h->gexec, g.b, t.b));
      }
      CK(cudaGraphLaunch(h->gexec, h->stream));
      h->launches += h->graph_nodes;
    } else {
      enqueue_iteration(h);
      CK(cudaGetLastError());
    }
  }
  CK(cudaEventRecord(h->ev_it1, h->stream));
  h->it_pending = true;
  h->iters_run += iters;
  return FREDOPT_OK;
}

int fredopt_end(fredopt_t h, float* w_out, float* dose_out, float* letd_out, fredopt_report* rep,
                uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!h->begun) return fail(h, FREDOPT_ERR_NOT_LOADED, "call fredopt_begin first");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  const int fb = list_blocks(h);
  if (h->it_pending) {
    float ms = 0.f;
    CK(cudaEventSynchronize(h->ev_it1));
    if (cudaEventElapsedTime(&ms, h->ev_it0, h->ev_it1) == cudaSuccess) h->device_ms += ms;
    h->it_pending = false;
  }
  // final double-float-accumulated product over every row
  rc = ready_y64(h);
  if (rc) return rc;
  float* dptr = nullptr;
  float* lptr = nullptr;
  if (dose_out || letd_out) {
    if (dev_ptr(flags)) {
      dptr = dose_out;
      lptr = letd_out;
    } else {
      CK(h->fout_a.ensure(std::max<int64_t>(1, h->V)));
      CK(h->fout_b.ensure(std::max<int64_t>(1, h->V)));
      dptr = dose_out ? h->fout_a.p : nullptr;
      lptr = letd_out ? h->fout_b.p : nullptr;
    }
  }
  if (dptr) CK(cudaMemsetAsync(dptr, 0, h->V * sizeof(float), s));
  if (lptr) CK(cudaMemsetAsync(lptr, 0, h->V * sizeof(float), s));
  FwdArgs fa = fwd_args(h, false, true);
  fa.x = h->w.p;
  fa.y64 = h->y64.p;
  fa.dose_out = dptr;
  fa.letd_out = lptr;
  run(h, 0, [&] { launch_forward(h->geo_full, h->fmt, EPI_FINAL, false, fa, h->tab, s); });
  double* pf = h->part.p + h->off_fin;
  run(h, 5, [&] { launch_final_check(fb, h->tab, h->y64.p, h->mask.p, h->mdd.p, h->mll.p, h->mdl.p, h->con_rows.p, h->n_con_rows, pf, s); });
  CK(cudaGetLastError());
  // staged: the solve state, then the check's partials
  constexpr size_t d_doubles = (sizeof(DevState) + sizeof(double) - 1) / sizeof(double);
  static_assert(d_doubles + 8 * 608 <= (size_t)kStageDoubles, "staging area");
  const double* hp = stage(h) + d_doubles;
  CK(cudaMemcpyAsync(stage(h), h->st.p, sizeof(DevState), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(stage(h) + d_doubles, pf, 8 * fb * sizeof(double), cudaMemcpyDeviceToHost, s));
  CK(copy_out(h, w_out, h->w.p, (size_t)h->n * sizeof(float), flags));
  if (!dev_ptr(flags)) {
    if (dose_out) CK(cudaMemcpyAsync(dose_out, h->fout_a.p, h->V * sizeof(float), cudaMemcpyDeviceToHost, s));
    if (letd_out) CK(cudaMemcpyAsync(letd_out, h->fout_b.p, h->V * sizeof(float), cudaMemcpyDeviceToHost, s));
  }
  rc = check_sticky(h);
  collect_timers(h);
  if (rc) return rc;
  DevState d;
  std::memcpy(&d, stage(h), sizeof(d));
  if (rep) {
    std::memset(rep, 0, sizeof(*rep));
    rep->iters = h->iters_run;
    rep->s = d.s;
    rep->accepted = d.accepted_total;
    rep->n_rows = h->n_rows_reach;
    rep->unreachable_rows = h->n_unreach;
    double nv = 0.0, f = 0.0;
    for (int b = 0; b < fb; ++b) {
      for (int q = 0; q < 6; ++q) rep->max_violation[q] = std::max(rep->max_violation[q], hp[8 * b + q]);
      nv += hp[8 * b + 6];
      f += hp[8 * b + 7];
    }
    rep->n_violated = (int64_t)nv;
    rep->objective = f;
    rep->beta0 = h->beta0;
    rep->device_ms = h->device_ms;
  }
  return FREDOPT_OK;
}

int fredopt_superiorize(fredopt_t h, const float* w0, int iters, double alpha, double relaxation,
                        const fredopt_params* params, float* w_out, float* dose_out,
                        float* letd_out, fredopt_report* rep, uint32_t flags) {
  int rc = fredopt_begin(h, w0, alpha, relaxation, params, flags);
  if (rc) return rc;
  rc = fredopt_iterate(h, iters);
  if (rc) return rc;
  return fredopt_end(h, w_out, dose_out, letd_out, rep, flags);
}

int fredopt_get_log(fredopt_t h, fredopt_log_entry* out, int max_entries) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!h->begun) return fail(h, FREDOPT_ERR_NOT_LOADED, "no solve begun");
  if (max_entries < 0 || (max_entries > 0 && !out)) return fail(h, FREDOPT_ERR_INVALID_ARG, "bad output");
  DeviceGuard dg(h->device);
  CK(cudaStreamSynchronize(h->stream));
  DevState d;
  CK(cudaMemcpy(&d, h->st.p, sizeof(DevState), cudaMemcpyDeviceToHost));
  const int cap = h->prm.log_capacity;
  if (cap <= 0) return 0;
  const int64_t k = d.k;
  const int64_t first = std::max<int64_t>(0, k - cap);
  const int cnt = (int)std::min<int64_t>(k - first, max_entries);
  std::vector<LogEntry> all(cap);
  CK(cudaMemcpy(all.data(), h->log.p, cap * sizeof(LogEntry), cudaMemcpyDeviceToHost));
  for (int i = 0; i < cnt; ++i) {
    const LogEntry& e = all[(first + i) % cap];
    out[i].k = e.k;
    out[i].s = e.s;
    out[i].accepted = e.accepted;
    out[i].n_violated = e.n_violated;
    out[i].beta = e.beta;
    out[i].f_start = e.f_start;
    out[i].f_end = e.f_end;
    out[i].gnorm = e.gnorm;
    out[i].max_violation = e.max_violation;
  }
  return cnt;
}

int fredopt_get_state(fredopt_t h, float* w, int64_t* k, int64_t* s, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!h->begun) return fail(h, FREDOPT_ERR_NOT_LOADED, "no solve begun");
  DeviceGuard dg(h->device);
  DevState d;
  CK(cudaMemcpyAsync(&d, h->st.p, sizeof(DevState), cudaMemcpyDeviceToHost, h->stream));
  if (w) CK(copy_out(h, w, h->w.p, (size_t)h->n * sizeof(float), flags));
  rc = check_sticky(h);
  if (rc) return rc;
  if (k) *k = d.k;
  if (s) *s = d.s;
  return FREDOPT_OK;
}

int fredopt_set_state(fredopt_t h, const float* w, int64_t k, int64_t s, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!h->begun) return fail(h, FREDOPT_ERR_NOT_LOADED, "call fredopt_begin first");
  if (!w || k < 0 || s < 0) return fail(h, FREDOPT_ERR_INVALID_ARG, "bad state");
  DeviceGuard dg(h->device);
  join_in(h);
  CK(cudaStreamSynchronize(h->stream));
  DevState d;
  CK(cudaMemcpy(&d, h->st.p, sizeof(DevState), cudaMemcpyDeviceToHost));
  d.k = k;
  d.s = s;
  d.done = 0u;
  CK(copy_in(h, h->w.p, w, (size_t)h->n * sizeof(float), flags));
  h->st_host = d;
  CK(cudaMemcpyAsync(h->st.p, &h->st_host, sizeof(DevState), cudaMemcpyHostToDevice, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return FREDOPT_OK;
}

int fredopt_forward(fredopt_t h, const float* w, float* dose_out, float* lw_out, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!w) return fail(h, FREDOPT_ERR_INVALID_ARG, "w is null");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  join_in(h);
  const float* xin = nullptr;
  rc = spot_in(h, w, flags, &xin);
  if (rc) return rc;
  if (!h->yall.p || h->yall.n < (size_t)std::max<int64_t>(1, h->V)) h->yall_zeroed = false;
  CK(h->yall.ensure(std::max<int64_t>(1, h->V)));
  if (!h->yall_zeroed) CK(cudaMemsetAsync(h->yall.p, 0, std::max<int64_t>(1, h->V) * sizeof(float2), s));
  h->yall_zeroed = true;
  FwdArgs fa = fwd_args(h, false);
  fa.x = xin;
  fa.y = h->yall.p;
  run(h, 0, [&] { launch_forward(h->geo_full, h->fmt, EPI_STORE, h->hint_fwd, fa, h->tab, s); });
  float *da = dose_out, *db = lw_out;
  if (!dev_ptr(flags)) {
    CK(h->fout_a.ensure(std::max<int64_t>(1, h->V)));
    CK(h->fout_b.ensure(std::max<int64_t>(1, h->V)));
    da = dose_out ? h->fout_a.p : nullptr;
    db = lw_out ? h->fout_b.p : nullptr;
  }
  launch_scatter_y(h->yall.p, h->perm ? h->voxel.p : nullptr, h->V, da, db, s);
  CK(cudaGetLastError());
  if (!dev_ptr(flags)) {
    if (dose_out) CK(cudaMemcpyAsync(dose_out, h->fout_a.p, h->V * sizeof(float), cudaMemcpyDeviceToHost, s));
    if (lw_out) CK(cudaMemcpyAsync(lw_out, h->fout_b.p, h->V * sizeof(float), cudaMemcpyDeviceToHost, s));
  }
  rc = check_sticky(h);
  collect_timers(h);
  return rc;
}

int fredopt_backward(fredopt_t h, const float* a_D, const float* a_L, float* u_out, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!u_out) return fail(h, FREDOPT_ERR_INVALID_ARG, "u_out is null");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  join_in(h);
  const float *pa = a_D, *pb = a_L;
  if (!dev_ptr(flags)) {
    CK(h->vin_a.ensure(std::max<int64_t>(1, h->V)));
    CK(h->vin_b.ensure(std::max<int64_t>(1, h->V)));
    if (a_D) CK(cudaMemcpyAsync(h->vin_a.p, a_D, h->V * sizeof(float), cudaMemcpyHostToDevice, s));
    if (a_L) CK(cudaMemcpyAsync(h->vin_b.p, a_L, h->V * sizeof(float), cudaMemcpyHostToDevice, s));
    pa = a_D ? h->vin_a.p : nullptr;
    pb = a_L ? h->vin_b.p : nullptr;
  }
  CK(h->ucoef.ensure(std::max<int64_t>(1, h->n_hot)));
  launch_scale_coef(h->n_hot, pa, pb, h->perm ? h->voxel.p : nullptr, h->fmt ? h->sD.p : nullptr,
                    h->fmt ? h->sL.p : nullptr, h->ucoef.p, s);
  BwdArgs ba = bwd_args(h, h->ucoef.p);
  run(h, 1, [&] { launch_backward(h->geo, h->fmt, h->hint_bwd, true, ba, s); });
  ColArgs ca = col_args(h);
  ca.out = spot_out(h, u_out, flags, h->gtmp);
  run(h, 3, [&] { launch_colfinish(h->geo, COL_OUT, ca, s); });
  CK(cudaGetLastError());
  if (ca.out != u_out) CK(copy_out(h, u_out, ca.out, (size_t)h->n * sizeof(float), flags));
  rc = check_sticky(h);
  collect_timers(h);
  return rc;
}

int fredopt_feasibility_step(fredopt_t h, const float* x, double relaxation, double prio_scale,
                             int norm, float* w_out, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!h->have_con) return fail(h, FREDOPT_ERR_NOT_LOADED, "no constraints set");
  if (!x || !w_out || !(relaxation > 0.0 && relaxation <= 2.0) || !(prio_scale > 0.0) ||
      (norm != FREDOPT_NORM_ALL && norm != FREDOPT_NORM_VIOLATED))
    return fail(h, FREDOPT_ERR_INVALID_ARG, "bad arguments");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  const Geometry& G = h->geo;
  join_in(h);
  const float* xin = nullptr;
  rc = spot_in(h, x, flags, &xin);
  if (rc) return rc;
  FwdArgs fa = fwd_args(h, true);
  fa.x = xin;
  fa.y = h->yw.p;
  run(h, 0, [&] { launch_forward(G, h->fmt, EPI_STORE, h->hint_fwd, fa, h->tab, s); });
  ConArgs k2 = con_args(h);
  run(h, 2, [&] { launch_constraints(G, h->tab, k2, s); });
  if (h->tab.n_con > 0) {
    BwdArgs bb = bwd_args(h, h->gam.p);
    run(h, 1, [&] { launch_backward(G, h->fmt, h->hint_bwd, true, bb, s); });
  }
  ColArgs cc = col_args(h);
  cc.w = xin;
  cc.w_out = spot_out(h, w_out, flags, h->xbuf, xin);
  cc.use_u = h->tab.n_con > 0 ? 1 : 0;
  cc.norm = norm;
  cc.lam = relaxation;
  cc.prio_scale = prio_scale;
  cc.in_solve = 0;
  cc.has_scale = norm != FREDOPT_NORM_VIOLATED ? 1 : 0;
  cc.scale = h->W_all > 0.0 ? relaxation * prio_scale / h->W_all : 0.0;
  run(h, 3, [&] { launch_colfinish(G, COL_PROJ, cc, s); });
  CK(cudaGetLastError());
  if (cc.w_out != w_out) CK(copy_out(h, w_out, cc.w_out, (size_t)h->n * sizeof(float), flags));
  rc = check_sticky(h);
  collect_timers(h);
  return rc;
}

int fredopt_sweep_step(fredopt_t h, const float* x, double relaxation, double prio_scale, int norm,
                       int n_blocks, float* w_out, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!x || !w_out) return fail(h, FREDOPT_ERR_INVALID_ARG, "null x or w_out");
  if (!(relaxation > 0.0 && relaxation <= 2.0)) return fail(h, FREDOPT_ERR_INVALID_ARG, "need 0 < relaxation <= 2");
  if (norm != FREDOPT_NORM_ALL && norm != FREDOPT_NORM_VIOLATED) return fail(h, FREDOPT_ERR_INVALID_ARG, "bad norm");
  if (n_blocks < 1 || n_blocks > FREDOPT_MAX_SWEEP_BLOCKS)
    return fail(h, FREDOPT_ERR_INVALID_ARG, "need 1 <= n_blocks <= FREDOPT_MAX_SWEEP_BLOCKS");
  if (h->begun && h->gexec && h->prm.sweep_blocks > 0 && h->sw->m != n_blocks)
    return fail(h, FREDOPT_ERR_INVALID_ARG, "the begun solve sweeps another number of blocks");
  DeviceGuard dg(h->device);
  join_in(h);
  // a begun solve that sweeps other blocks (in plain launches or a batch graph)
  // keeps its own: this call's are built aside and freed at its end
  struct Aside {
    fredopt_t h;
    std::unique_ptr<Sweep> own;
    ~Aside() {
      if (!own) return;
      cudaStreamSynchronize(h->stream);
      h->sw = std::move(own);
    }
  } aside{h, nullptr};
  if (h->begun && h->prm.sweep_blocks > 0 && h->sw->m != n_blocks) {
    aside.own = std::move(h->sw);
    h->sw.reset(new Sweep());
  }
  rc = build_sweep(h, n_blocks);
  if (rc) return rc;
  const float* xin = nullptr;
  rc = spot_in(h, x, flags, &xin);
  if (rc) return rc;
  float* dst = spot_out(h, w_out, flags, h->gtmp);
  enqueue_sweep(h, xin, 0, relaxation, prio_scale, norm, 0, dst);
  CK(cudaGetLastError());
  if (dst != w_out) CK(copy_out(h, w_out, dst, (size_t)h->n * sizeof(float), flags));
  rc = check_sticky(h);
  collect_timers(h);
  return rc;
}

int fredopt_objective(fredopt_t h, const float* x, double* f_out, float* grad_out, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!x) return fail(h, FREDOPT_ERR_INVALID_ARG, "x is null");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  const Geometry& G = h->geo;
  join_in(h);
  const float* xin = nullptr;
  rc = spot_in(h, x, flags, &xin);
  if (rc) return rc;
  double* part_f = h->part.p + h->off_f;
  FwdArgs fa = fwd_args(h, true);
  fa.x = xin;
  fa.y = h->yw.p;
  fa.r_out = h->r.p;
  fa.part = part_f;
  run(h, 0, [&] { launch_forward(G, h->fmt, EPI_OBJ, h->hint_fwd, fa, h->tab, s); });
  BwdArgs ba = bwd_args(h, h->r.p);
  run(h, 1, [&] { launch_backward(G, h->fmt, h->hint_bwd, h->obj_dose, ba, s); });
  ColArgs ca = col_args(h);
  ca.out = spot_out(h, grad_out, flags, h->gtmp);
  ca.part = h->part.p + h->off_g;
  run(h, 3, [&] { launch_colfinish(G, COL_GRAD, ca, s); });
  // claimed tiles leave tens of thousands of partials: summed to kFinishBlocks first
  int np = n_parts(G, fa);
  const double* pf = part_f;
  if (np > 1024) {
    pf = h->part.p + h->off_stage;
    launch_sum_slices(part_f, np, h->part.p + h->off_stage, s);
    np = kFinishBlocks;
  }
  CK(cudaGetLastError());
  CK(cudaMemcpyAsync(stage(h), pf, np * sizeof(double), cudaMemcpyDeviceToHost, s));
  if (grad_out && ca.out != grad_out) CK(copy_out(h, grad_out, ca.out, (size_t)h->n * sizeof(float), flags));
  rc = check_sticky(h);
  collect_timers(h);
  if (rc) return rc;
  if (f_out) {
    double f = f_empty(h);
    for (int i = 0; i < np; ++i) f += stage(h)[i];
    *f_out = f;
  }
  return FREDOPT_OK;
}

int fredopt_volume_stats(fredopt_t h, const float* w, uint32_t flags, int n_req, fredopt_volume_request* req) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (n_req < 0 || n_req > FREDOPT_VOLUME_MAX_REQUESTS || (n_req > 0 && !req))
    return fail(h, FREDOPT_ERR_INVALID_ARG, "need 0 <= n_req <= FREDOPT_VOLUME_MAX_REQUESTS and req");
  VolArgs va{};
  SelArgs sa{};
  std::vector<float> edges;
  std::vector<double> fracs;
  std::vector<int> sel_req;
  int n_bins = 0;
  for (int i = 0; i < n_req; ++i) {
    const fredopt_volume_request& r = req[i];
    if (r.quantity < FREDOPT_Q_DOSE || r.quantity > FREDOPT_Q_LETD)
      return fail(h, FREDOPT_ERR_INVALID_ARG, "quantity must be FREDOPT_Q_DOSE, _CDL or _LETD");
    if (r.struct_bit < 0 || r.struct_bit > 31) return fail(h, FREDOPT_ERR_INVALID_ARG, "struct_bit must be 0..31");
    if (r.n_bins < 0 || r.n_fracs < 0) return fail(h, FREDOPT_ERR_INVALID_ARG, "negative n_bins or n_fracs");
    if (r.n_bins > 0 && (!r.edges || !r.counts)) return fail(h, FREDOPT_ERR_INVALID_ARG, "edges or counts is null");
    if (r.n_fracs > 0 && (!r.fracs || !r.at_volume))
      return fail(h, FREDOPT_ERR_INVALID_ARG, "fracs or at_volume is null");
    if (n_bins + (int64_t)r.n_bins > FREDOPT_VOLUME_MAX_BINS)
      return fail(h, FREDOPT_ERR_INVALID_ARG, "more than FREDOPT_VOLUME_MAX_BINS bins in total");
    if ((int64_t)fracs.size() + r.n_fracs > FREDOPT_VOLUME_MAX_FRACS)
      return fail(h, FREDOPT_ERR_INVALID_ARG, "more than FREDOPT_VOLUME_MAX_FRACS fractions in total");
    for (int b = 0; b <= r.n_bins && r.n_bins > 0; ++b) {
      if (std::isnan(r.edges[b])) return fail(h, FREDOPT_ERR_INVALID_ARG, "NaN edge");
      if (b > 0 && r.edges[b] < r.edges[b - 1]) return fail(h, FREDOPT_ERR_INVALID_ARG, "edges decrease");
    }
    for (int q = 0; q < r.n_fracs; ++q)
      if (!(r.fracs[q] > 0.0 && r.fracs[q] <= 1.0)) return fail(h, FREDOPT_ERR_INVALID_ARG, "fraction outside (0, 1]");
    va.q[i] = r.quantity;
    va.bit[i] = r.struct_bit;
    va.nb[i] = r.n_bins;
    va.eoff[i] = (int32_t)edges.size();
    va.boff[i] = n_bins;
    if (r.n_bins > 0) edges.insert(edges.end(), r.edges, r.edges + r.n_bins + 1);
    n_bins += r.n_bins;
    for (int q = 0; q < r.n_fracs; ++q) {
      const int j = (int)fracs.size();
      sa.q[j] = r.quantity;
      sa.bit[j] = r.struct_bit;
      sel_req.push_back(i);
      fracs.push_back(r.fracs[q]);
    }
    va.any_bits |= 1u << r.struct_bit;
  }
  if (n_req == 0) return FREDOPT_OK;
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  join_in(h);
  rc = final_pass_y64(h, w, flags, true);
  if (rc) return rc;

  // scratch: inputs (edges | fractions), then results (counts | n_vox |
  // selection slots), then digit histograms; one copy each way
  const int n_sel = (int)fracs.size();
  const size_t o_fracs = align256(std::max<size_t>(1, edges.size()) * sizeof(float));
  const size_t o_counts = o_fracs + align256(std::max(1, n_sel) * sizeof(double));
  const size_t o_nvox = o_counts + align256(std::max(1, n_bins) * sizeof(unsigned long long));
  const size_t o_slot = o_nvox + align256(n_req * sizeof(unsigned long long));
  const size_t o_hist = o_slot + align256(std::max(1, n_sel) * sizeof(SelSlot));
  const size_t total = o_hist + align256(std::max(1, n_sel) * 256 * sizeof(uint32_t));
  CK(h->vol_buf.ensure(total));
  uint8_t* base = h->vol_buf.p;
  std::vector<uint8_t> io(std::max(o_counts, o_hist - o_counts));
  if (!edges.empty()) std::memcpy(io.data(), edges.data(), edges.size() * sizeof(float));
  if (n_sel) std::memcpy(io.data() + o_fracs, fracs.data(), n_sel * sizeof(double));
  CK(cudaMemsetAsync(base + o_counts, 0, total - o_counts, s));
  CK(cudaMemcpyAsync(base, io.data(), o_counts, cudaMemcpyHostToDevice, s));

  va.y64 = h->y64.p;
  va.mask = h->mask.p;
  va.rows = h->con_rows.p;  // every structure voxel is a streamed row
  va.n_rows = h->n_con_rows;
  va.c = h->tab.c;
  va.n_req = n_req;
  va.n_edges = (int)edges.size();
  va.n_bins = n_bins;
  va.edges = reinterpret_cast<const float*>(base);
  va.counts = reinterpret_cast<unsigned long long*>(base + o_counts);
  va.n_vox = reinterpret_cast<unsigned long long*>(base + o_nvox);
  run(h, 5, [&] { launch_vol_hist(h->geo, va, s); });
  CK(cudaGetLastError());
  if (n_sel > 0) {
    for (int j = 0; j < n_sel; ++j) sa.req[j] = sel_req[j];
    sa.y64 = h->y64.p;
    sa.mask = h->mask.p;
    sa.rows = h->con_rows.p;
    sa.n_rows = h->n_con_rows;
    sa.c = h->tab.c;
    sa.any_bits = va.any_bits;
    sa.n_sel = n_sel;
    sa.fracs = reinterpret_cast<const double*>(base + o_fracs);
    sa.n_vox = va.n_vox;
    sa.hist = reinterpret_cast<uint32_t*>(base + o_hist);
    sa.st = reinterpret_cast<SelSlot*>(base + o_slot);
    run(h, 5, [&] { launch_vol_select(h->geo, sa, s); });
    h->launches += kVolSelectLaunches - 1;
    CK(cudaGetLastError());
  }
  CK(cudaMemcpyAsync(io.data(), base + o_counts, o_hist - o_counts, cudaMemcpyDeviceToHost, s));
  rc = check_sticky(h);
  collect_timers(h);
  if (rc) return rc;
  const unsigned long long* counts = reinterpret_cast<const unsigned long long*>(io.data());
  const unsigned long long* nvox = reinterpret_cast<const unsigned long long*>(io.data() + (o_nvox - o_counts));
  const SelSlot* slots = reinterpret_cast<const SelSlot*>(io.data() + (o_slot - o_counts));
  int j = 0;
  for (int i = 0; i < n_req; ++i) {
    fredopt_volume_request& r = req[i];
    r.n_voxels = (int64_t)nvox[i];
    for (int b = 0; b < r.n_bins; ++b) r.counts[b] = (int64_t)counts[va.boff[i] + b];
    for (int q = 0; q < r.n_fracs; ++q, ++j)
      r.at_volume[q] = nvox[i] > 0 ? key_to_float(slots[j].prefix) : std::numeric_limits<float>::quiet_NaN();
  }
  return FREDOPT_OK;
}

int fredopt_quantity_map(fredopt_t h, const float* w, int quantity, float* out, uint32_t flags) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (!out) return fail(h, FREDOPT_ERR_INVALID_ARG, "out is null");
  if (quantity < FREDOPT_Q_DOSE || quantity > FREDOPT_Q_LETD)
    return fail(h, FREDOPT_ERR_INVALID_ARG, "quantity must be FREDOPT_Q_DOSE, _CDL or _LETD");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  join_in(h);
  rc = final_pass_y64(h, w, flags, false);
  if (rc) return rc;
  float* dst = out;
  if (!dev_ptr(flags)) {
    CK(h->fout_a.ensure(std::max<int64_t>(1, h->V)));
    dst = h->fout_a.p;
  }
  run(h, 5, [&] { launch_vol_map(h->geo, h->y64.p, h->perm ? h->voxel.p : nullptr, h->V, quantity, h->tab.c, dst, s); });
  CK(cudaGetLastError());
  if (!dev_ptr(flags) && h->V > 0)
    CK(cudaMemcpyAsync(out, dst, h->V * sizeof(float), cudaMemcpyDeviceToHost, s));
  rc = check_sticky(h);
  collect_timers(h);
  return rc;
}

int fredopt_get_sizes(fredopt_t h, int64_t* n_vox, int64_t* n_spots, int64_t* nnz, int64_t* n_rows,
                      int64_t* nnz_rows) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (n_vox) *n_vox = h->V;
  if (n_spots) *n_spots = h->n;
  if (nnz) *nnz = h->nnz;
  if (n_rows) *n_rows = h->n_hot;
  if (nnz_rows) *nnz_rows = h->nnz_hot;
  return FREDOPT_OK;
}

int fredopt_get_storage(fredopt_t h, int* col_index_bytes, int* row_index_bytes, int* val_bytes) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (col_index_bytes) *col_index_bytes = h->col16.p ? 2 : 4;
  if (row_index_bytes) *row_index_bytes = h->crow16.p ? 2 : 4;
  if (val_bytes) *val_bytes = value_bytes(h->fmt);
  return FREDOPT_OK;
}

int fredopt_get_rows(fredopt_t h, int64_t* voxel, uint32_t* mask) {
  int rc = need_loaded(h);
  if (rc) return rc;
  DeviceGuard dg(h->device);
  if (voxel) {
    if (h->perm) {
      CK(cudaMemcpy(voxel, h->voxel.p, h->n_hot * sizeof(int64_t), cudaMemcpyDeviceToHost));
    } else {
      for (int64_t i = 0; i < h->n_hot; ++i) voxel[i] = i;
    }
  }
  if (mask && h->n_hot) CK(cudaMemcpy(mask, h->mask.p, h->n_hot * sizeof(uint32_t), cudaMemcpyDeviceToHost));
  return FREDOPT_OK;
}

int fredopt_get_csc(fredopt_t h, int64_t* col_ptr, int32_t* row, float* D_val, float* L_val) {
  int rc = need_loaded(h);
  if (rc) return rc;
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  if (col_ptr) CK(cudaMemcpyAsync(col_ptr, h->cp.p, (h->n + 1) * sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  if (row && h->nnz_hot) CK(cudaMemcpyAsync(row, h->crow.p, h->nnz_hot * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  if ((D_val || L_val) && h->nnz_hot) {
    DBuf<float> a, b;
    CK(a.alloc(h->nnz_hot));
    CK(b.alloc(h->nnz_hot));
    launch_dequant_csc(h->fmt, h->cp.p, h->n, h->crow.p, h->DTv.p, h->LTv.p, h->fmt ? h->sD.p : nullptr,
                       h->fmt ? h->sL.p : nullptr, a.p, b.p, s);
    CK(cudaGetLastError());
    if (D_val) CK(cudaMemcpyAsync(D_val, a.p, h->nnz_hot * sizeof(float), cudaMemcpyDeviceToHost, s));
    if (L_val) CK(cudaMemcpyAsync(L_val, b.p, h->nnz_hot * sizeof(float), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
  }
  CK(cudaStreamSynchronize(s));
  return FREDOPT_OK;
}

int fredopt_get_moments(fredopt_t h, double* dd, double* ll, double* dl) {
  int rc = need_loaded(h);
  if (rc) return rc;
  DeviceGuard dg(h->device);
  CK(cudaStreamSynchronize(h->stream));
  if (h->n_hot == 0) return FREDOPT_OK;
  if (dd) CK(cudaMemcpy(dd, h->mdd.p, h->n_hot * sizeof(double), cudaMemcpyDeviceToHost));
  if (ll) CK(cudaMemcpy(ll, h->mll.p, h->n_hot * sizeof(double), cudaMemcpyDeviceToHost));
  if (dl) CK(cudaMemcpy(dl, h->mdl.p, h->n_hot * sizeof(double), cudaMemcpyDeviceToHost));
  return FREDOPT_OK;
}

int fredopt_set_timing(fredopt_t h, int enable) {
  if (!h) return FREDOPT_ERR_INVALID_ARG;
  DeviceGuard dg(h->device);
  collect_timers(h);
  h->timing = enable != 0;
  for (int i = 0; i < FREDOPT_KCLASS_N; ++i) {
    h->kms[i] = 0.0;
    h->klaunch[i] = 0;
  }
  h->launches = 0;
  return FREDOPT_OK;
}

int fredopt_get_timing(fredopt_t h, double* ms, int64_t* launches) {
  if (!h) return FREDOPT_ERR_INVALID_ARG;
  DeviceGuard dg(h->device);
  collect_timers(h);
  for (int i = 0; i < FREDOPT_KCLASS_N; ++i) {
    if (ms) ms[i] = h->kms[i];
    if (launches) launches[i] = h->klaunch[i];
  }
  return FREDOPT_OK;
}

int64_t fredopt_launch_count(fredopt_t h) { return h ? h->launches : -1; }

int fredopt_kernel_arch(int device, int* fwd_binary, int* bwd_binary, int* ptx_version) {
  int cur = 0;
  if (cudaGetDevice(&cur) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) {
    cudaGetLastError();
    return FREDOPT_ERR_CUDA;
  }
  const cudaError_t e = kernel_arch(fwd_binary, bwd_binary, ptx_version);
  cudaSetDevice(cur);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return FREDOPT_ERR_CUDA;
  }
  return FREDOPT_OK;
}

int fredopt_check_wait(fredopt_t h, int arrive, int spins, float* elapsed_ms) {
  if (!h) return FREDOPT_ERR_INVALID_ARG;
  if (spins < 0) return fail(h, FREDOPT_ERR_INVALID_ARG, "spins must be >= 0");
  DeviceGuard dg(h->device);
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return fail(h, FREDOPT_ERR_CUDA, "event create");
  }
  cudaEventRecord(e0, h->stream);
  launch_wait_check(arrive, spins, h->st.p, h->stream);
  cudaError_t e = cudaGetLastError();
  cudaEventRecord(e1, h->stream);
  const int rc = e != cudaSuccess ? cuda_fail(h, e, "wait check launch") : check_sticky(h);
  if (elapsed_ms) {
    float ms = 0.0f;
    if (cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) ms = -1.0f;
    *elapsed_ms = ms;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return rc;
}

int fredopt_get_tuning(fredopt_t h, int64_t* row_cost, int64_t* chunk_cost) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (row_cost) *row_cost = h->row_cost;
  if (chunk_cost) *chunk_cost = h->chunk_cost;
  return FREDOPT_OK;
}

int fredopt_autotune(fredopt_t h, int reps, int64_t* row_cost, int64_t* chunk_cost) {
  int rc = need_loaded(h);
  if (rc) return rc;
  if (reps < 1 || h->timing) return fail(h, FREDOPT_ERR_INVALID_ARG, "reps >= 1, timing off");
  DeviceGuard dg(h->device);
  cudaStream_t s = h->stream;
  const Geometry& G = h->geo;
  // inputs: w of the solve if one is begun, else ones; coefficients 1
  if (!h->begun) {
    std::vector<float> ones(h->n, 1.0f);
    CK(cudaMemcpyAsync(h->xbuf.p, ones.data(), h->n * sizeof(float), cudaMemcpyHostToDevice, s));
    CK(cudaStreamSynchronize(s));
  }
  const float* x = h->begun ? h->w.p : h->xbuf.p;
  launch_scale_coef(h->n_hot, nullptr, nullptr, nullptr, nullptr, nullptr, h->gam.p, s);
  cudaEvent_t e0, e1;
  CK(cudaEventCreate(&e0));
  CK(cudaEventCreate(&e1));
  auto time_ms = [&](auto&& launch) -> float {
    launch();  // warm-up
    float best = 1e30f;
    for (int i = 0; i < reps; ++i) {
      cudaEventRecord(e0, s);
      launch();
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      best = std::min(best, ms);
    }
    return best;
  };
  FwdArgs fa = fwd_args(h, true);
  fa.x = x;
  fa.y = h->yw.p;
  int64_t best_row = h->row_cost;
  float best_f = 1e30f;
  for (int64_t c : kRowCosts) {
    if ((rc = set_fwd_schedule(h, c))) break;
    const float t = time_ms([&] { launch_forward(G, h->fmt, EPI_STORE, h->hint_fwd, fa, h->tab, s); });
    if (t < best_f) { best_f = t; best_row = c; }
  }
  BwdArgs ba = bwd_args(h, h->gam.p);
  int64_t best_chunk = h->chunk_cost;
  float best_b = 1e30f;
  for (int64_t c : kChunkCosts) {
    if (rc || (rc = set_bwd_schedule(h, c))) break;
    const float t = time_ms([&] { launch_backward(G, h->fmt, h->hint_bwd, true, ba, s); });
    if (t < best_b) { best_b = t; best_chunk = c; }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (rc) return rc;
  if ((rc = set_fwd_schedule(h, best_row))) return rc;
  if ((rc = set_bwd_schedule(h, best_chunk))) return rc;
  rc = check_sticky(h);
  if (rc) return rc;
  if (row_cost) *row_cost = best_row;
  if (chunk_cost) *chunk_cost = best_chunk;
  return FREDOPT_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ batches

struct fredopt_batch {
  int device = 0;
  cudaStream_t root = nullptr;
  std::vector<fredopt_t> hs;
  std::vector<int> nodes;
  cudaGraph_t graph = nullptr;      // one iteration of every plan
  cudaGraphExec_t exec = nullptr;
  int depth = 1;                    // iterations of every plan in graph_k
  cudaGraph_t graph_k = nullptr;
  cudaGraphExec_t exec_k = nullptr;
  cudaEvent_t fork = nullptr, done = nullptr, t0 = nullptr, t1 = nullptr;
  std::vector<cudaEvent_t> joins;
  double ms = 0.0;
  bool pending = false;
};

namespace {
void batch_free(fredopt_batch* b) {
  if (b->root) cudaStreamSynchronize(b->root);
  if (b->exec) cudaGraphExecDestroy(b->exec);
  if (b->graph) cudaGraphDestroy(b->graph);
  if (b->exec_k) cudaGraphExecDestroy(b->exec_k);
  if (b->graph_k) cudaGraphDestroy(b->graph_k);
  for (cudaEvent_t e : b->joins) cudaEventDestroy(e);
  for (cudaEvent_t e : {b->fork, b->done, b->t0, b->t1})
    if (e) cudaEventDestroy(e);
  if (b->root) cudaStreamDestroy(b->root);
  delete b;
}
}  // namespace

extern "C" {

int fredopt_batch_create(fredopt_batch_t* out, const fredopt_t* handles, int n) {
  return fredopt_batch_create_depth(out, handles, n, 1);
}

int fredopt_batch_create_depth(fredopt_batch_t* out, const fredopt_t* handles, int n, int depth) {
  if (!out || !handles || n < 1 || depth < 1 || depth > FREDOPT_BATCH_MAX_DEPTH) return FREDOPT_ERR_INVALID_ARG;
  *out = nullptr;
  const int dev = handles[0] ? handles[0]->device : -1;
  for (int i = 0; i < n; ++i) {
    fredopt_t h = handles[i];
    if (!h || !h->loaded || !h->begun || h->device != dev || h->timing) return FREDOPT_ERR_NOT_LOADED;
    for (int j = 0; j < i; ++j)
      if (handles[j] == h || handles[j]->stream == h->stream) return FREDOPT_ERR_INVALID_ARG;
  }
  DeviceGuard dg(dev);
  fredopt_batch* b = new fredopt_batch();
  b->device = dev;
  b->hs.assign(handles, handles + n);
  auto bad = [&](cudaError_t e) {
    batch_free(b);
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? FREDOPT_ERR_OOM : FREDOPT_ERR_CUDA;
  };
  cudaError_t e;
  if ((e = cudaStreamCreateWithFlags(&b->root, cudaStreamNonBlocking)) != cudaSuccess) return bad(e);
  for (cudaEvent_t* ev : {&b->fork, &b->done})
    if ((e = cudaEventCreateWithFlags(ev, cudaEventDisableTiming)) != cudaSuccess) return bad(e);
  if ((e = cudaEventCreate(&b->t0)) != cudaSuccess || (e = cudaEventCreate(&b->t1)) != cudaSuccess) return bad(e);
  b->joins.resize(n, nullptr);
  for (int i = 0; i < n; ++i) {
    if ((e = cudaEventCreateWithFlags(&b->joins[i], cudaEventDisableTiming)) != cudaSuccess) return bad(e);
    if ((e = cudaStreamSynchronize(handles[i]->stream)) != cudaSuccess) return bad(e);
  }
  // `iters` iterations of every plan as parallel branches of one graph (each
  // branch runs its plan's iterations in order, exactly as alone)
  auto capture = [&](int iters, cudaGraph_t* g, cudaGraphExec_t* x) -> cudaError_t {
    cudaError_t ce = cudaStreamBeginCapture(b->root, cudaStreamCaptureModeThreadLocal);
    if (ce != cudaSuccess) return ce;
    cudaEventRecord(b->fork, b->root);
    for (int i = 0; i < n; ++i) {
      fredopt_t h = handles[i];
      cudaStreamWaitEvent(h->stream, b->fork, 0);
      const int64_t before = h->launches;
      for (int k = 0; k < iters; ++k) enqueue_iteration(h);
      if (iters == 1) b->nodes.push_back((int)(h->launches - before));
      h->launches = before;
      cudaEventRecord(b->joins[i], h->stream);
      cudaStreamWaitEvent(b->root, b->joins[i], 0);
    }
    ce = cudaStreamEndCapture(b->root, g);
    if (ce != cudaSuccess) {
      *g = nullptr;
      return ce;
    }
    return cudaGraphInstantiate(x, *g, 0);
  };
  if ((e = capture(1, &b->graph, &b->exec)) != cudaSuccess) return bad(e);
  b->depth = depth;
  if (depth > 1 && (e = capture(depth, &b->graph_k, &b->exec_k)) != cudaSuccess) return bad(e);
  *out = b;
  return FREDOPT_OK;
}

int fredopt_batch_iterate(fredopt_batch_t b, int iters) {
  if (!b || iters < 0) return FREDOPT_ERR_INVALID_ARG;
  if (iters == 0) return FREDOPT_OK;
  DeviceGuard dg(b->device);
  if (b->pending) {
    float ms = 0.f;
    cudaEventSynchronize(b->t1);
    if (cudaEventElapsedTime(&ms, b->t0, b->t1) == cudaSuccess) b->ms += ms;
    b->pending = false;
  }
  for (fredopt_t h : b->hs) {  // order after any work the caller queued on the plans
    cudaEventRecord(h->ev_join, h->stream);
    cudaStreamWaitEvent(b->root, h->ev_join, 0);
  }
  cudaEventRecord(b->t0, b->root);
  // whole graphs of `depth` iterations, then single iterations
  const int nk = b->exec_k ? iters / b->depth : 0;
  for (int i = 0; i < nk; ++i)
    if (cudaGraphLaunch(b->exec_k, b->root) != cudaSuccess) {
      cudaGetLastError();
      return FREDOPT_ERR_CUDA;
    }
  for (int i = nk * b->depth; i < iters; ++i)
    if (cudaGraphLaunch(b->exec, b->root) != cudaSuccess) {
      cudaGetLastError();
      return FREDOPT_ERR_CUDA;
    }
  cudaEventRecord(b->t1, b->root);
  b->pending = true;
  cudaEventRecord(b->done, b->root);
  for (size_t i = 0; i < b->hs.size(); ++i) {
    fredopt_t h = b->hs[i];
    cudaStreamWaitEvent(h->stream, b->done, 0);  // later calls on the plan see the iterations
    h->iters_run += iters;
    h->launches += (int64_t)iters * b->nodes[i];
  }
  return FREDOPT_OK;
}

int fredopt_batch_sync(fredopt_batch_t b, double* device_ms) {
  if (!b) return FREDOPT_ERR_INVALID_ARG;
  DeviceGuard dg(b->device);
  if (cudaStreamSynchronize(b->root) != cudaSuccess) {
    cudaGetLastError();
    return FREDOPT_ERR_CUDA;
  }
  if (b->pending) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, b->t0, b->t1) == cudaSuccess) b->ms += ms;
    b->pending = false;
  }
  if (device_ms) *device_ms = b->ms;
  for (fredopt_t h : b->hs) {
    if (*err_word(h)) return FREDOPT_ERR_TIMEOUT;
  }
  return FREDOPT_OK;
}

int fredopt_batch_destroy(fredopt_batch_t b) {
  if (!b) return FREDOPT_ERR_INVALID_ARG;
  DeviceGuard dg(b->device);
  batch_free(b);
  return FREDOPT_OK;
}

int fredopt_superiorize_batch(const fredopt_t* handles, int n, const float* const* w0, int iters, double alpha,
                              double relaxation, const fredopt_params* params, float* const* w_out,
                              float* const* dose_out, float* const* letd_out, fredopt_report* reps,
                              uint32_t flags) {
  if (!handles || !w0 || n < 1) return FREDOPT_ERR_INVALID_ARG;
  fredopt_params p;
  if (params) p = *params;
  else fredopt_default_params(&p);
  p.use_graphs = 0;  // the batch graph replaces the per-plan graphs
  for (int i = 0; i < n; ++i) {
    const int rc = fredopt_begin(handles[i], w0[i], alpha, relaxation, &p, flags);
    if (rc) return rc;
  }
  fredopt_batch_t b = nullptr;
  int rc = fredopt_batch_create_depth(&b, handles, n, std::max(1, std::min(iters, FREDOPT_BATCH_DEPTH)));
  if (rc) return rc;
  rc = fredopt_batch_iterate(b, iters);
  if (!rc) rc = fredopt_batch_sync(b, nullptr);
  fredopt_batch_destroy(b);
  if (rc) return rc;
  for (int i = 0; i < n; ++i) {
    rc = fredopt_end(handles[i], w_out ? w_out[i] : nullptr, dose_out ? dose_out[i] : nullptr,
                     letd_out ? letd_out[i] : nullptr, reps ? &reps[i] : nullptr, flags);
    if (rc) return rc;
  }
  return FREDOPT_OK;
}

}  // extern "C"

namespace fo {
cudaStream_t handle_stream(fredopt_t h) { return h ? h->stream : nullptr; }
int handle_device(fredopt_t h) { return h ? h->device : -1; }
}  // namespace fo

extern "C" {

}  // extern "C"
