// The library's host code (fredopt_api.cu) over a CUDA runtime and kernels that
// are stand-ins on the CPU, for what the host does when a runtime call or a
// device-side wait fails.  "Device" memory is host memory; kernels compute
// nothing beyond the totals that the load reads.  Compiled by tests/test_host_failures_cpu.py.
#include <cstdlib>
#include <map>

#include "../paper_2509_20012_gb300/csrc/fredopt_api.cu"

namespace {
std::map<void*, size_t> g_blocks;
size_t g_used = 0, g_peak = 0, g_limit = ~(size_t)0;
int g_fail_waits = 0;      // forward products whose bounded wait gives up
int g_fail_captures = 0;   // cudaStreamBeginCapture calls that fail
int g_capturing = 0, g_stray_external = 0;
int g_sweep_blocks = 0;
const void *g_sweep_pos = nullptr, *g_captured_pos = nullptr;
int g_long_checks = 0;     // products whose stated array length is not that of every array
void check_length(int64_t n, const void* idx, size_t ib, const void* d, const void* l, int fmt) {
  const size_t vb = fmt == 0 ? 4 : 2;
  for (auto [p, b] : {std::pair{idx, ib}, std::pair{d, vb}, std::pair{l, vb}})
    if ((size_t)n * b > g_blocks[const_cast<void*>(p)]) ++g_long_checks;
}
long long g_nnz_hot = 0;
}  // namespace

extern "C" {
size_t fake_used() { return g_used; }
size_t fake_peak() { return g_peak; }
void fake_limit(size_t bytes) { g_limit = bytes; g_peak = g_used; }
void fake_fail_waits(int n) { g_fail_waits = n; }
void fake_fail_captures(int n) { g_fail_captures = n; }
int fake_stray_external() { return g_stray_external; }
int fake_sweep_blocks() {  // blocks swept since the last call
  const int n = g_sweep_blocks;
  g_sweep_blocks = 0;
  return n;
}
void fake_capture_pos() { g_captured_pos = g_sweep_pos; }  // the tables of the last sweep
int fake_captured_alive() { return g_blocks.count(const_cast<void*>(g_captured_pos)); }
int fake_long_checks() { return g_long_checks; }
size_t fake_bar_offset(int n_x_pad) { return fo::fwd_bar_offset(n_x_pad); }

// ---- CUDA runtime
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_used + n > g_limit) return cudaErrorMemoryAllocation;
  *p = std::malloc(n);
  std::memset(*p, 0xee, n);
  g_blocks[*p] = n;
  g_used += n;
  g_peak = std::max(g_peak, g_used);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  g_used -= g_blocks[p];
  g_blocks.erase(p);
  return cudaSuccess;  // not handed out again: a stale pointer shows
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { std::memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 1 << 27; return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  static size_t next = 16;  // a stream is a number
  *s = reinterpret_cast<cudaStream_t>(next++);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  if (g_fail_captures > 0) {
    --g_fail_captures;
    return cudaErrorStreamCaptureUnsupported;
  }
  g_capturing = 1;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  g_capturing = 0;
  *g = reinterpret_cast<cudaGraph_t>(1);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(1); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned f) {
  if (f == cudaEventRecordExternal && !g_capturing) ++g_stray_external;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.0f; return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  *x = reinterpret_cast<cudaGraphExec_t>(1);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) { *n = 0; return cudaSuccess; }
cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType*) { return cudaSuccess; }
cudaError_t cudaGraphEventRecordNodeGetEvent(cudaGraphNode_t, cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaGraphExecEventRecordNodeSetEvent(cudaGraphExec_t, cudaGraphNode_t, cudaEvent_t) { return cudaSuccess; }
}  // extern "C"

// ---- kernels
namespace fo {
int init_kernels(Geometry* g, int) {
  *g = Geometry{2, 1024, 2, 64, 256, 8, 64, 256, 8, 256, 4, (size_t)227 * 1024};
  return 0;
}
cudaError_t kernel_arch(int*, int*, int*) { return cudaSuccess; }
bool forward_uses_smem(const Geometry&, int) { return true; }
int forward_grid(const Geometry& g, int) { return g.fwd_blocks; }
int col_grid(const Geometry& g, int) { return g.col_blocks; }
int con_grid(const Geometry& g, int64_t) { return g.row_blocks; }
void launch_forward(const Geometry&, int fmt, int, bool, const FwdArgs& a, const Tables&, cudaStream_t) {
  check_length(a.n_elems, a.col16 ? (const void*)a.col16 : a.col, a.col16 ? 2 : 4, a.Dv, a.Lv, fmt);
  if (g_fail_waits > 0) {
    --g_fail_waits;
    *a.st->err |= 1;
  }
}
void launch_backward(const Geometry&, int fmt, bool, bool, const BwdArgs& a, cudaStream_t) {
  check_length(a.n_elems, a.row16 ? (const void*)a.row16 : a.row, a.row16 ? 2 : 4, a.Dv, a.Lv, fmt);
}
void launch_colfinish(const Geometry&, int, const ColArgs&, cudaStream_t) {}
void launch_constraints(const Geometry&, const Tables&, const ConArgs&, cudaStream_t) {}
void launch_beta_table(double*, long long, double, double, cudaStream_t) {}
void launch_finish(int, const double*, int, const double*, int, const double*, int, DevState*, double*, const double*,
                   long long, bool, cudaStream_t) {}
void launch_count_rows(int grid, const Tables&, const uint32_t*, const double*, const double*, const double*,
                       const int64_t*, int64_t, double* part, cudaStream_t) {
  std::memset(part, 0, 3 * grid * sizeof(double));
}
void launch_scatter_y(const float2*, const int64_t*, int64_t, float*, float*, cudaStream_t) {}
void launch_apply_step(int64_t, int, float*, const float*, float2*, const float2*, const DevState*, cudaStream_t) {}
void launch_row_objective(const Geometry&, const Tables&, const float2*, const uint32_t*, const float*, const float*,
                          int64_t, float2*, double*, cudaStream_t) {}
void launch_final_check(int, const Tables&, const double2*, const uint32_t*, const double*, const double*,
                        const double*, const int64_t*, int64_t, double*, cudaStream_t) {}
void launch_check_spots(const float*, int32_t, double* part, cudaStream_t) {
  for (int b = 0; b < kSpotSlices; ++b) part[2 * b + 1] = (double)kNoSpot;
}
void launch_sum_slices(const double*, int, double*, cudaStream_t) {}
size_t row_order_scratch(int64_t n) { return (size_t)n / 256 + 8; }
void launch_rows_count(const int64_t* rp, const uint32_t* mask, int64_t n, int64_t nnz, bool, int64_t*, RowTotals* t,
                       cudaStream_t) {
  for (int64_t i = 0; i < n; ++i) {
    t->c[0] += 1;  // every row streamed, with nonzeros
    t->c[5] += mask[i] != 0u;
  }
  t->c[3] = g_nnz_hot = nnz;
}
void launch_rows_place(const int64_t*, const uint32_t*, int64_t, bool, const int64_t*, const RowTotals*, int64_t*,
                       int64_t*, uint32_t*, int64_t*, float*, float*, cudaStream_t) {}
void launch_load_rows(int, bool, bool, const LoadRowsArgs&, cudaStream_t) {}
void launch_tiles(const TileArgs&, cudaStream_t) {}
void launch_csc_columns(const int64_t*, int32_t n, int64_t, int64_t* cp, int32_t* col_chunk, cudaStream_t) {
  cp[n] = g_nnz_hot;
  col_chunk[n] = n;
}
void launch_chunk_fill(const int64_t*, const int32_t*, int32_t, int64_t, int64_t*, cudaStream_t) {}
CscShape csc_shape(const Geometry& g, int, int64_t n_rows, int32_t n_cols, int64_t) {
  CscShape q{};
  q.n_rows = n_rows;
  q.n_cols = n_cols;
  q.n_strip = g.n_sms;
  return q;
}
void launch_csc_count(const CscShape&, size_t, const int64_t*, const int32_t*, const uint16_t*, const int64_t*,
                      int32_t*, int32_t*, cudaStream_t) {}
void launch_csc_colsum(const int32_t*, int, int32_t, int64_t*, cudaStream_t) {}
void launch_csc_offsets(int32_t*, int, int32_t, const int64_t*, cudaStream_t) {}
void launch_csc_fill(const CscShape&, int, const int64_t*, const int32_t*, const uint16_t*, const void*, const void*,
                     const int64_t*, const int32_t*, int32_t*, int32_t*, void*, void*, cudaStream_t) {}
void launch_dequant_csc(int, const int64_t*, int32_t, const int32_t*, const void*, const void*, const float*,
                        const float*, float*, float*, cudaStream_t) {}
void launch_scale_coef(int64_t, const float*, const float*, const int64_t*, const float*, const float*, float2*,
                       cudaStream_t) {}
void launch_narrow_rows(const int32_t*, int64_t, uint16_t*, int32_t*, unsigned int*, cudaStream_t) {}
void launch_narrow_rows_wide(const int32_t*, int64_t, int32_t*, int32_t*, unsigned int*, unsigned int, cudaStream_t) {}
void launch_wait_check(int arrive, int, DevState* st, cudaStream_t) {
  if (!arrive) *st->err |= 1;
}
void launch_sweep_start(int, const float*, const float*, int, float*, DevState*, cudaStream_t) {}
void launch_sweep_pos(const int64_t*, const int32_t*, int32_t, const int64_t*, int, int64_t*, cudaStream_t) {}
int sweep_weight_slices(int64_t) { return 1; }
void launch_sweep_weights(const Tables&, const int64_t*, int64_t, int64_t, int, const uint32_t*, const double*,
                          const double*, const double*, double*, double*, cudaStream_t) {}
void launch_sweep_rows(int fmt, double, const SweepArgs& a, cudaStream_t) {
  check_length(a.n_elems, a.col16 ? (const void*)a.col16 : a.col, a.col16 ? 2 : 4, a.rD, a.rL, fmt);
  check_length(a.n_csc, a.row, 4, a.Dv, a.Lv, fmt);
  if (a.i0 == 0) g_sweep_pos = a.pos0;
  ++g_sweep_blocks;
}
void launch_sweep_con(const Tables&, const SweepArgs&, cudaStream_t) {}
void launch_sweep_lengths(const int64_t*, int32_t, int n, double* out, cudaStream_t) {
  std::memset(out, 0, 2 * n * sizeof(double));
}
void launch_sweep_cols(int, double, double, const SweepArgs&, cudaStream_t) {}
void launch_sweep_finish(const Geometry&, int, const float*, float*, int, DevState*, LogEntry*, cudaStream_t) {}
size_t vol_hist_smem(const VolArgs&) { return 0; }
void launch_vol_hist(const Geometry&, const VolArgs&, cudaStream_t) {}
void launch_vol_select(const Geometry&, const SelArgs&, cudaStream_t) {}
void launch_vol_map(const Geometry&, const double2*, const int64_t*, int64_t, int, double, float*, cudaStream_t) {}
}  // namespace fo
