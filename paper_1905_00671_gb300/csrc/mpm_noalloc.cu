// mpm_noalloc.cu -- mpm_bin_noalloc: the cell binning and (cell, index)
// ordering of material points, for callers that cannot allocate device memory.
//
// Who needs it: code that may not call cudaMalloc at the point where it bins
// points -- for example a solver embedded in a host application that owns all
// device memory through its own pool and gives libraries no allocator, or a
// latency-critical loop where the implicit device synchronisation of
// cudaMalloc / cudaFree is not acceptable.  The caller passes the positions and
// the two output arrays; the per-cell counters live in the fixed array below.
//
// The scratch array is a file-scope __device__ variable: every GPU that loads
// this library holds it (about 2 MiB) until the process exits, and every call
// on that GPU shares it.  Host code cannot use the array's name as a device
// address; the first call on each device looks the address up with
// cudaGetSymbolAddress (with that device current) and keeps it.  Because that
// first call does this set-up (and synchronises), it should be made before any
// stream capture.  Every call, not only the first, copies an error word to the
// host and waits for its stream before it returns.  The counters a call needs
// at zero are cleared by the call; two calls that overlap on the GPU
// (different streams, or host threads that do not order them) race on the
// shared array and give wrong results.
#include <math.h>
#include <string.h>

#include <atomic>

#include "mpm_internal.cuh"

namespace upmpm {
namespace {

constexpr int64_t NOALLOC_MAX_CELLS = 1 << 18;   // 262,144 cells
constexpr int NOALLOC_MAX_DEVICES = 64;
constexpr int NA_HEAD = 64;                      // the error word, alone on its lines
constexpr int NA_SCAN = 4096;                    // cells per block of the scan
// layout: the error word, then [0, C] counts (one clear covers both), padded to
// whole scan blocks, then [0, C] cell starts
constexpr int64_t NOALLOC_INTS = NA_HEAD + 2 * (NOALLOC_MAX_CELLS + NA_SCAN);

static __device__ __align__(256) int32_t g_noalloc_scratch[NOALLOC_INTS];

std::atomic<int32_t *> g_scratch_ptr[NOALLOC_MAX_DEVICES];

int scratch_for_current_device(int32_t **out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return MPM_ERR_CUDA;
  int32_t *p = g_scratch_ptr[dev].load(std::memory_order_acquire);
  if (!p) {
    void *addr = nullptr;
    if (cudaGetSymbolAddress(&addr, g_noalloc_scratch) != cudaSuccess || !addr) return MPM_ERR_CUDA;
    p = static_cast<int32_t *>(addr);
    g_scratch_ptr[dev].store(p, std::memory_order_release);
  }
  *out = p;
  return MPM_OK;
}

// floor(d / h) as the correctly rounded quotient gives it.  d * (1 / h) is
// within 2^-50 of that quotient, relatively, so its floor is the same one unless
// an integer lies that close; only then (and for zeros, infinities and NaN, where the
// comparison fails, and next to zero, where a quotient is too small for a relative
// bound) is the division made.  The FP64 pipe does 2 operations a cycle and SM
// and a division costs about ten.
__device__ __forceinline__ double cell_floor(double d, double h, double inv) {
  const double q = d * inv;
  if (fabs(q - rint(q)) > fma(0x1p-50, fabs(q), 0x1p-1000)) return floor(q);
  return floor(__ddiv_rn(d, h));
}

template <int D>
__global__ void k_na_keys(GridP g, double inv, int64_t n, const double *__restrict__ x, int32_t *__restrict__ cell,
                          int32_t *__restrict__ count, int32_t *__restrict__ err) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= n) return;
  int c[3] = {0, 0, 0};
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const double cf = cell_floor(__dsub_rn(x[p * D + k], g.org[k]), g.h, inv);
    if (!(cf >= 0.0) || !(cf <= (double)(g.nc[k] - 1))) {
      atomicOr(err, 1);
      cell[p] = -1;
      return;
    }
    c[k] = (int)cf;
  }
  const int32_t id = (int32_t)cell_index(g, c[0], c[1], c[2]);
  cell[p] = id;
  atomicAdd(&count[id], 1);
}

// Exclusive scan of count[0..m) into start[0..m], NA_SCAN cells to a block of
// 1024 threads.  A block adds up everything before its own cells itself
// (coalesced 16-byte loads from L2: 64 a thread at most, for the last block of the
// largest grid), so that no block waits for another and one launch is enough.
// One block that walked a run of cells per thread took 15 us of latency at 20k cells
// with every other SM idle.
__global__ void __launch_bounds__(1024) k_na_scan(const int32_t *__restrict__ count, int64_t m,
                                                  int32_t *__restrict__ start, const int32_t *__restrict__ err) {
  __shared__ int32_t wsum[32], wpre[32];
  if (*err) return;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t seg = blockIdx.x * (int64_t)NA_SCAN;
  const int4 *c4 = reinterpret_cast<const int4 *>(count);
  int32_t before = 0;
#pragma unroll 4
  for (int64_t i = t; i < seg / 4; i += 1024) {
    const int4 v = c4[i];
    before += v.x + v.y + v.z + v.w;
  }
  const int64_t i0 = seg + 4 * t;
  int32_t v[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = i0 + k < m ? count[i0 + k] : 0;
  const int32_t own = v[0] + v[1] + v[2] + v[3];
  int32_t inc = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  before = __reduce_add_sync(0xffffffffu, before);
  if (lane == 31) wsum[warp] = inc;
  if (lane == 0) wpre[warp] = before;
  __syncthreads();
  int32_t run = __reduce_add_sync(0xffffffffu, wpre[lane]) +
                __reduce_add_sync(0xffffffffu, lane < warp ? wsum[lane] : 0) + inc - own;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (i0 + k < m) start[i0 + k] = run;
    run += v[k];
    if (i0 + k == m - 1) start[m] = run;
  }
}

// each point takes a slot of its cell by counting the cell's counter down
__global__ void k_na_scatter(int64_t n, const int32_t *__restrict__ cell, const int32_t *__restrict__ start,
                             int32_t *__restrict__ count, int64_t *__restrict__ order,
                             const int32_t *__restrict__ err) {
  const int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= n || *err) return;
  const int32_t c = cell[p];
  order[start[c] + atomicSub(&count[c], 1) - 1] = p;
}

// The points of each cell in increasing order, 8 lanes to a cell: a cell of up
// to 8 points is read once, each lane counts the smaller ones and writes its own to
// that place; larger cells are sorted in place by odd-even transposition, whose
// pairs the lanes share.
__global__ void k_na_sort(int64_t ncells, const int32_t *__restrict__ start, int64_t *order,
                          const int32_t *__restrict__ err) {
  const int64_t c = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
  if (c >= ncells || *err) return;                 // all 8 lanes of a cell alike
  const int lane = threadIdx.x & 31, l = lane & 7;
  const unsigned mask = 0xffu << (lane & 24);
  const int32_t b = start[c];
  const int32_t n = start[c + 1] - b;
  if (n < 2) return;
  int64_t *o = order + b;
  if (n <= 8) {
    const int32_t v = l < n ? (int32_t)o[l] : INT32_MAX;
    int r = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) r += __shfl_sync(mask, v, j, 8) < v;
    __syncwarp(mask);
    if (l < n) o[r] = v;
    return;
  }
  for (int32_t s = 0; s < n; ++s) {
    for (int32_t i = (s & 1) + 2 * l; i + 1 < n; i += 16) {
      const int64_t u = o[i], w = o[i + 1];
      if (u > w) {
        o[i] = w;
        o[i + 1] = u;
      }
    }
    __syncwarp(mask);
  }
}

}  // namespace
}  // namespace upmpm

using namespace upmpm;

extern "C" int mpm_bin_noalloc(const mpm_grid *grid, int64_t n, const double *x_dev,
                               int32_t *cell_dev, int64_t *order_dev, void *stream) {
  if (!grid || n < 0 || (n > 0 && (!x_dev || !cell_dev || !order_dev))) return MPM_ERR_BAD_ARG;
  if (grid->dim != 2 && grid->dim != 3) return MPM_ERR_BAD_ARG;
  if (!(grid->h > 0.0) || n > INT32_MAX) return MPM_ERR_BAD_ARG;
  // Each axis is bounded before the product is formed, so the product of at
  // most three factors <= 2^18 cannot overflow int64 and a grid whose cell
  // count would wrap is rejected rather than indexed.  Only the cell fields
  // of GridP are used here.
  GridP g{};
  g.d = grid->dim;
  g.ncells = 1;
  for (int k = 0; k < 3; ++k) {
    const bool used = k < g.d;
    if (used && grid->ncell[k] < 1) return MPM_ERR_BAD_ARG;
    if (used && grid->ncell[k] > NOALLOC_MAX_CELLS) return MPM_ERR_TOO_LARGE;
    g.nc[k] = used ? grid->ncell[k] : 1;
    g.org[k] = used ? grid->origin[k] : 0.0;
    g.ncells *= g.nc[k];
  }
  g.h = grid->h;
  if (g.ncells > NOALLOC_MAX_CELLS) return MPM_ERR_TOO_LARGE;
  int32_t *scr = nullptr;
  int rc = scratch_for_current_device(&scr);
  if (rc) return rc;
  cudaStream_t st = (cudaStream_t)stream;
  const int64_t C = g.ncells;
  int32_t *err = scr, *count = scr + NA_HEAD, *start = count + (NOALLOC_MAX_CELLS + NA_SCAN);
  // everything this call reads before writing starts at zero
  if (cudaMemsetAsync(scr, 0, sizeof(int32_t) * (NA_HEAD + C + 1), st) != cudaSuccess) return MPM_ERR_CUDA;
  // The later kernels read the error word themselves and do nothing once it is
  // set, so the host waits once, at the end, and not between them.  With that, one
  // clear for three and the kernels above, binning 80k points took 72 -> 50 us.
  if (n > 0) {
    const int nbk = (int)((n + 255) / 256);
    const double inv = 1.0 / g.h;
    if (g.d == 2) k_na_keys<2><<<nbk, 256, 0, st>>>(g, inv, n, x_dev, cell_dev, count, err);
    else k_na_keys<3><<<nbk, 256, 0, st>>>(g, inv, n, x_dev, cell_dev, count, err);
    k_na_scan<<<(int)((C + NA_SCAN - 1) / NA_SCAN), 1024, 0, st>>>(count, C, start, err);
    k_na_scatter<<<nbk, 256, 0, st>>>(n, cell_dev, start, count, order_dev, err);
    k_na_sort<<<(int)((8 * C + 255) / 256), 256, 0, st>>>(C, start, order_dev, err);
  }
  int32_t herr = 0;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(&herr, err, sizeof(int32_t), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return MPM_ERR_CUDA;
  return herr ? MPM_ERR_OUT_OF_GRID : MPM_OK;
}
