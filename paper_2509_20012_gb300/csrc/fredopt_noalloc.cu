// Transposed product u = D^T a_D + L^T a_L over caller-owned device arrays
// without any device allocation.
//
// Some callers of this library cannot allocate device memory at the point
// where they need the product: a host application that hands every byte of
// the GPU to its own memory pool (so a stray cudaMalloc would fail or
// fragment the pool), or a latency-critical loop in which cudaMalloc and
// cudaFree are avoided because they can synchronise the device and stall
// work already queued.  This entry point needs no handle and no allocation:
// its scratch (per-chunk partial sums) is one fixed file-scope device array,
// held by every GPU that loads the library until the process exits.
//
// The work is split like the library's transposed product: each column is cut
// into chunks of kNaChunk nonzeros, every chunk is summed by one warp in a
// fixed order, and the chunk sums of a column are added in chunk order, so
// the result is deterministic.
#include "fredopt.h"

#include <cuda_runtime.h>

#include <cstdint>
#include <mutex>

namespace {

constexpr int kNaChunk = 4096;          // nonzeros per chunk
constexpr int kNaMaxCols = 65536;       // largest n_cols accepted
constexpr int kNaMaxChunks = 1 << 20;   // largest number of chunks accepted
constexpr size_t kNaScratchBytes = (size_t)kNaMaxChunks * sizeof(float);

// The scratch: chunk sums (float[kNaMaxChunks]).  4 MiB.  Every call rewrites
// the parts it reads, so nothing has to start at zero.
static __device__ __align__(256) unsigned char g_na_scratch[kNaScratchBytes];

constexpr int kMaxDevices = 64;
std::mutex g_na_mutex;
void* g_na_addr[kMaxDevices] = {nullptr};

// Device address of the scratch on the current device, looked up once per
// device (cudaGetSymbolAddress with that device current) and kept for the
// life of the process.  A cudaDeviceReset reloads the module, so the kept
// address is no longer valid after one.
cudaError_t scratch_address(void** out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lk(g_na_mutex);
  if (!g_na_addr[dev]) {
    void* p = nullptr;
    e = cudaGetSymbolAddress(&p, g_na_scratch);
    if (e != cudaSuccess) return e;
    g_na_addr[dev] = p;
  }
  *out = g_na_addr[dev];
  return cudaSuccess;
}

__device__ __forceinline__ int64_t clamp_ptr(int64_t v, int64_t nnz) {
  return v < 0 ? 0 : (v > nnz ? nnz : v);
}

// Column j's chunks take the places slot(j) .. slot(j) + count - 1 of the
// scratch, slot(j) = col_ptr[j] / kNaChunk + j: ceil(length / kNaChunk) is at
// most one more than the chunk boundaries a column spans, so the places of two
// columns never overlap, and nnz / kNaChunk + n_cols places are enough.  No scan
// is needed (a one-block scan of 30000 columns took 54 us); one pass over the
// columns leaves every place's column in it (-1: no chunk), where the place's
// warp reads it before it writes the sum.
struct NaCol {
  int64_t s, e;  // the column's nonzeros (pointers clamped to [0, nnz], empty if they do not ascend)
  int32_t slot;
  __device__ NaCol(const int64_t* col_ptr, int64_t nnz, int32_t j) {
    s = clamp_ptr(col_ptr[j], nnz);
    e = clamp_ptr(col_ptr[j + 1], nnz);
    if (e < s) e = s;
    slot = (int32_t)(s / kNaChunk) + j;
  }
  __device__ int32_t count() const { return (int32_t)((e - s + kNaChunk - 1) / kNaChunk); }
};

__global__ void __launch_bounds__(256) k_na_slots(const int64_t* __restrict__ col_ptr, int32_t n_cols, int64_t nnz,
                                                  int32_t n_slots, int32_t* __restrict__ slot_col) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_cols) return;
  const NaCol c(col_ptr, nnz, j);
  const int32_t used = c.slot + c.count();
  const int32_t next = j + 1 < n_cols ? (int32_t)(c.e / kNaChunk) + j + 1 : n_slots;
  for (int32_t g = c.slot; g < used; ++g) slot_col[g] = j;
  for (int32_t g = used; g < next; ++g) slot_col[g] = -1;
}

// One warp per chunk: sum of D_ij a_D[i] + L_ij a_L[i] over the chunk, in
// entry order per lane.  The loads of kNaUnroll steps, then their gathers, are in
// flight together (without a branch between them), and the grid has a warp per
// place, so that the SMs even out uneven chunks: 7.7e7 nonzeros 218 -> 156 us
// (12 bytes per nonzero take 137; one step in flight and eight CTAs per SM
// striding over the chunks were the 218).
constexpr int kNaUnroll = 6;
template <bool HAVE_D, bool HAVE_L>
__global__ void __launch_bounds__(256, 6) k_na_chunks(const int64_t* __restrict__ col_ptr,
                                                      const int32_t* __restrict__ row, const float* __restrict__ Dv,
                                                      const float* __restrict__ Lv, const float* __restrict__ aD,
                                                      const float* __restrict__ aL, int64_t n_rows, int32_t n_cols,
                                                      int64_t nnz, int32_t n_slots, float* part) {
  const int lane = threadIdx.x & 31;
  const int32_t g = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  if (g >= n_slots) return;
  const int32_t j = reinterpret_cast<const int32_t*>(part)[g];  // k_na_slots left the column here
  // (pointers that do not ascend leave places unset: anything may be in them)
  if (j < 0 || j >= n_cols) return;
  const NaCol c(col_ptr, nnz, j);
  if (g < c.slot || g >= c.slot + c.count()) return;
  const int64_t s = c.s + (int64_t)(g - c.slot) * kNaChunk;
  const int n = (int)(s + kNaChunk < c.e ? kNaChunk : c.e - s);
  float acc = 0.0f;
  const int32_t* __restrict__ rp = row + s;
  const float* __restrict__ dp = Dv + s;
  const float* __restrict__ lp = Lv + s;
  // whole steps without branches (rows out of range read entry 0 of the
  // coefficients and contribute nothing), then the rest one by one
  int i = lane;
  for (; i + 32 * (kNaUnroll - 1) < n; i += 32 * kNaUnroll) {
    int32_t r[kNaUnroll];
    float d[kNaUnroll], l[kNaUnroll], x[kNaUnroll], y[kNaUnroll];
    bool ok[kNaUnroll];
#pragma unroll
    for (int k = 0; k < kNaUnroll; ++k) {
      r[k] = __ldcs(rp + i + 32 * k);
      if (HAVE_D) d[k] = __ldcs(dp + i + 32 * k);
      if (HAVE_L) l[k] = __ldcs(lp + i + 32 * k);
    }
#pragma unroll
    for (int k = 0; k < kNaUnroll; ++k) {
      ok[k] = r[k] >= 0 && r[k] < n_rows;
      const int32_t q = ok[k] ? r[k] : 0;
      if (HAVE_D) x[k] = __ldg(aD + q);
      if (HAVE_L) y[k] = __ldg(aL + q);
    }
#pragma unroll
    for (int k = 0; k < kNaUnroll; ++k) {
      if (HAVE_D) acc = ok[k] ? fmaf(d[k], x[k], acc) : acc;
      if (HAVE_L) acc = ok[k] ? fmaf(l[k], y[k], acc) : acc;
    }
  }
  for (; i < n; i += 32) {
    const int32_t r = __ldcs(rp + i);
    if (r < 0 || r >= n_rows) continue;  // never read outside the coefficient arrays
    if (HAVE_D) acc = fmaf(__ldcs(dp + i), __ldg(aD + r), acc);
    if (HAVE_L) acc = fmaf(__ldcs(lp + i), __ldg(aL + r), acc);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (lane == 0) part[g] = acc;  // every lane's read of part[g] came before the first shuffle
}

// u_j = sum of the chunk sums of column j, in chunk order.
__global__ void __launch_bounds__(256) k_na_columns(const int64_t* __restrict__ col_ptr, const float* __restrict__ part,
                                                    int32_t n_cols, int64_t nnz, float* __restrict__ u) {
  const int32_t j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n_cols) return;
  const NaCol c(col_ptr, nnz, j);
  const int32_t end = c.slot + c.count();
  float s = 0.0f;
  for (int32_t g = c.slot; g < end; ++g) s += part[g];
  u[j] = s;
}

}  // namespace

extern "C" int fredopt_backward_noalloc(int64_t n_rows, int32_t n_cols, int64_t nnz, const int64_t* col_ptr,
                                        const int32_t* row, const float* D_val, const float* L_val,
                                        const float* a_D, const float* a_L, float* u_out, void* cuda_stream) {
  if (n_rows < 0 || n_cols < 1 || nnz < 0) return FREDOPT_ERR_SHAPE;
  if (n_cols > kNaMaxCols || nnz / kNaChunk + n_cols > kNaMaxChunks) return FREDOPT_ERR_SHAPE;
  if (!col_ptr || !u_out || (nnz > 0 && (!row || !D_val || !L_val))) return FREDOPT_ERR_INVALID_ARG;
  void* base = nullptr;
  if (scratch_address(&base) != cudaSuccess) {
    cudaGetLastError();
    return FREDOPT_ERR_CUDA;
  }
  float* part = reinterpret_cast<float*>(base);
  const int32_t n_slots = (int32_t)(nnz / kNaChunk) + n_cols;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(cuda_stream);
  const unsigned col_grid = (unsigned)((n_cols + 255) / 256);
  k_na_slots<<<col_grid, 256, 0, s>>>(col_ptr, n_cols, nnz, n_slots, reinterpret_cast<int32_t*>(part));
  if (n_rows == 0) a_D = a_L = nullptr;  // no coefficient to read
  auto* chunks = a_D ? (a_L ? k_na_chunks<true, true> : k_na_chunks<true, false>)
                     : (a_L ? k_na_chunks<false, true> : k_na_chunks<false, false>);
  chunks<<<(unsigned)((n_slots + 7) / 8), 256, 0, s>>>(col_ptr, row, D_val, L_val, a_D, a_L, n_rows, n_cols, nnz, n_slots, part);
  k_na_columns<<<col_grid, 256, 0, s>>>(col_ptr, part, n_cols, nnz, u_out);
  if (cudaGetLastError() != cudaSuccess) return FREDOPT_ERR_CUDA;
  return FREDOPT_OK;
}
