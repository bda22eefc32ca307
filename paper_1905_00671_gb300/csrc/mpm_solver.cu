// mpm_solver.cu -- linear algebra of the Newton step (Eq. jacobian-system-
// stabilized-ppp):  J dX = -R  on the block-CSR Jacobian.
//
// The system is scaled symmetrically, D J D y = -D R with D_ii = |J_ii|^{-1/2},
// which brings the momentum rows (stiffness ~ 1e7) and the mass rows (~ 1e-7)
// to unit diagonal so that the Krylov residual weighs both balance laws; then
// right-preconditioned restarted FGMRES with classical Gram-Schmidt applied
// twice (in FP64 on single systems: where the first pass needs the second) solves
// it.  The Hessenberg matrix and the Givens rotations live
// in device memory (FP64); the host reads one scalar per iteration.  Vectors
// and matrix values are in the precision T of the solve: FP64, or FP32 in the
// mixed mode (the Newton residual around it stays FP64).  Reductions use a
// fixed grid and tree (deterministic) and sum each thread's part in T before
// the FP64 block sum.  No tensor cores: the work is sparse.
#include <math.h>

#include <algorithm>
#include <vector>

#include "mpm_internal.cuh"

namespace upmpm {

namespace {

constexpr int TPB = 256;
constexpr int NPART = 304;  // partial sums per reduction (2 x 152 SMs)
constexpr int PSTR = 129;   // stride of the per-block partial sums (restart <= 128)
constexpr int ORTH_TPB = 1024;     // threads per block of the Gram-Schmidt update ...
constexpr int64_t ORTH_BIG = 1 << 20;  // ... on systems of at least this many unknowns
// FP64 Gram-Schmidt: the second pass of classical Gram-Schmidt runs when the
// first left less than this fraction of the new vector's norm (it then lost
// more digits than a second pass needs to restore; otherwise one pass keeps
// the basis orthogonal to round-off: on the oracle's Jacobian of a slope piece
// the first pass left 0.2-0.5 of the norm and the basis orthogonal to 4e-15
// with one pass).  FP32 keeps both passes always.
constexpr double REORTH_THETA = 0.01;
inline int nblk(int64_t n, int tpb = TPB) { return (int)((n + tpb - 1) / tpb); }

__device__ inline double block_sum(double v) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  const int nw = (blockDim.x + 31) >> 5;
  v = (threadIdx.x < nw) ? sh[threadIdx.x] : 0.0;
  if (wid == 0)
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;  // valid in thread 0
}

// ---------------------------------------------------------------- scan
constexpr int SCAN_T = 1024, SCAN_I = 4, SCAN_CHUNK = SCAN_T * SCAN_I;

__device__ inline int block_excl_scan(int v, int *total) {
  __shared__ int sh[32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[wid] = x;
  __syncthreads();
  if (wid == 0) {
    int s = sh[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    sh[lane] = s;
  }
  __syncthreads();
  const int before = wid > 0 ? sh[wid - 1] : 0;
  *total = sh[31];
  __syncthreads();
  return before + x - v;
}

__global__ void k_scan_blocks(const int32_t *__restrict__ in, int32_t *__restrict__ out, int64_t n,
                              int32_t *__restrict__ blk) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_I;
  int v[SCAN_I], s = 0;
  for (int i = 0; i < SCAN_I; ++i) {
    v[i] = (base + i < n) ? in[base + i] : 0;
    s += v[i];
  }
  int total;
  int run = block_excl_scan(s, &total);
  for (int i = 0; i < SCAN_I; ++i) {
    if (base + i < n) out[base + i] = run;
    run += v[i];
  }
  if (threadIdx.x == 0) blk[blockIdx.x] = total;
}

__global__ void k_scan_top(int32_t *__restrict__ blk, int nb) {
  const int base = threadIdx.x * SCAN_I;  // one block; nb <= SCAN_CHUNK
  int v[SCAN_I], s = 0;
  for (int i = 0; i < SCAN_I; ++i) {
    v[i] = (base + i < nb) ? blk[base + i] : 0;
    s += v[i];
  }
  int total;
  int run = block_excl_scan(s, &total);
  for (int i = 0; i < SCAN_I; ++i) {
    if (base + i < nb) blk[base + i] = run;
    run += v[i];
  }
}

__global__ void k_scan_add(int32_t *__restrict__ out, int64_t n, const int32_t *__restrict__ blk,
                           const int32_t *__restrict__ in, double *total_out) {
  const int64_t base = (int64_t)blockIdx.x * SCAN_CHUNK + (int64_t)threadIdx.x * SCAN_I;
  const int32_t add = blk[blockIdx.x];
  for (int i = 0; i < SCAN_I; ++i)
    if (base + i < n) {
      out[base + i] += add;
      if (base + i == n - 1) slot_write(total_out, (double)out[base + i] + (double)in[base + i]);
    }
}

// ---------------------------------------------------------------- vectors
template <typename T>
__global__ void k_dot_partial(const T *__restrict__ x, const T *__restrict__ y, int64_t n,
                              double *__restrict__ part) {
  pdl_enter();
  T acc = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    acc += x[i] * y[i];
  const double s = block_sum((double)acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

__global__ void k_reduce(const double *__restrict__ part, int np, double *__restrict__ out) {
  pdl_enter();
  double acc = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) acc += part[i];
  acc = block_sum(acc);
  if (threadIdx.x == 0) out[0] = acc;
}

// The same into a mapped result word, with the device error word beside it.
__global__ void k_reduce_post(const double *__restrict__ part, int np, const int *__restrict__ err, double *out,
                              double *out_err) {
  pdl_enter();
  double acc = 0.0;
  for (int i = threadIdx.x; i < np; i += blockDim.x) acc += part[i];
  acc = block_sum(acc);
  if (threadIdx.x == 0) {
    slot_write(out_err, (double)*err);
    slot_write(out, acc);
  }
}

__global__ void k_post_err(const int *__restrict__ err, double *out) { slot_write(out, (double)*err); }

template <typename T>
__global__ void k_scale_copy(T *__restrict__ y, const T *__restrict__ x, const double *s, int64_t n) {
  pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = x[i] * (T)s[0];
}

template <typename T>
__global__ void k_residual_vec(T *__restrict__ y, const T *__restrict__ b, int64_t n) {  // y = b - y
  pdl_enter();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = b[i] - y[i];
}

// ---------------------------------------------------------------- scaling
__device__ inline int find_diag(const int32_t *__restrict__ row_ptr, const int32_t *__restrict__ col,
                                int64_t a) {
  int lo = row_ptr[a], hi = row_ptr[a + 1] - 1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1;
    const int cm = col[mid];
    if (cm == a) return mid;
    if (cm < a) lo = mid + 1; else hi = mid - 1;
  }
  return -1;
}

template <int NB, typename T>
__global__ void k_diag_scale(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, const T *__restrict__ val,
                             T *__restrict__ dsc, T *__restrict__ dsci) {
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  const int e = find_diag(row_ptr, col, a);
  for (int r = 0; r < NB; ++r) {
    const double d = e >= 0 ? fabs((double)val[(int64_t)e * NB * NB + r * NB + r]) : 0.0;
    dsc[a * NB + r] = (T)(d > 0.0 ? 1.0 / sqrt(d) : 1.0);
    dsci[a * NB + r] = (T)(d > 0.0 ? sqrt(d) : 1.0);
  }
}

template <typename T>
__global__ void k_scale_rhs(int64_t n, const double *__restrict__ R, const T *__restrict__ dsc,
                            T *__restrict__ rhs) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) rhs[i] = (T)(-(double)dsc[i] * R[i]);
}

template <typename T>
__global__ void k_add(int64_t n, double *__restrict__ X, const T *__restrict__ x) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) X[i] += (double)x[i];
}

template <typename T>
__global__ void k_mul(int64_t n, T *__restrict__ z, const T *__restrict__ s) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) z[i] *= s[i];
}

// ---------------------------------------------------------------- block Jacobi
// D (D J D)_aa^{-1}: from a vector of the scaled system to the unscaled unknowns
template <int NB, typename T>
__global__ void k_block_jacobi(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                               const int32_t *__restrict__ col, const T *__restrict__ val,
                               const T *__restrict__ dsc, T *__restrict__ dinv, int *err) {
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  const int e = find_diag(row_ptr, col, a);
  double A[NB][NB], B[NB][NB];
  for (int i = 0; i < NB; ++i)
    for (int j = 0; j < NB; ++j) {
      A[i][j] = e >= 0 ? (double)val[(int64_t)e * NB * NB + i * NB + j] * (double)(dsc[a * NB + i] * dsc[a * NB + j])
                       : (i == j ? 1.0 : 0.0);
      B[i][j] = i == j ? 1.0 : 0.0;
    }
  bool ok = true;  // Gauss-Jordan with partial pivoting
  for (int k = 0; k < NB; ++k) {
    int piv = k;
    double best = fabs(A[k][k]);
    for (int i = k + 1; i < NB; ++i)
      if (fabs(A[i][k]) > best) { best = fabs(A[i][k]); piv = i; }
    if (!(best > 1e-300)) { ok = false; break; }
    if (piv != k)
      for (int j = 0; j < NB; ++j) {
        double t = A[k][j]; A[k][j] = A[piv][j]; A[piv][j] = t;
        t = B[k][j]; B[k][j] = B[piv][j]; B[piv][j] = t;
      }
    const double inv = 1.0 / A[k][k];
    for (int j = 0; j < NB; ++j) { A[k][j] *= inv; B[k][j] *= inv; }
    for (int i = 0; i < NB; ++i) {
      if (i == k) continue;
      const double f = A[i][k];
      if (f == 0.0) continue;
      for (int j = 0; j < NB; ++j) { A[i][j] -= f * A[k][j]; B[i][j] -= f * B[k][j]; }
    }
  }
  if (!ok) {
    atomicOr(err, DE_SINGULAR);
    for (int i = 0; i < NB; ++i)
      for (int j = 0; j < NB; ++j) B[i][j] = i == j ? 1.0 : 0.0;
  }
  for (int i = 0; i < NB; ++i)
    for (int j = 0; j < NB; ++j) dinv[a * NB * NB + i * NB + j] = (T)((double)dsc[a * NB + i] * B[i][j]);
}

template <int NB, typename T>
__global__ void k_bj_apply(int64_t nnodes, const T *__restrict__ dinv, const T *__restrict__ x,
                           T *__restrict__ y) {
  pdl_enter();
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  T xv[NB];
  for (int j = 0; j < NB; ++j) xv[j] = x[a * NB + j];
  for (int i = 0; i < NB; ++i) {
    T s = 0;
    for (int j = 0; j < NB; ++j) s += dinv[a * NB * NB + i * NB + j] * xv[j];
    y[a * NB + i] = s;
  }
}

// ---------------------------------------------------------------- SpMV
// NB values of a block row, or of a node's x.  FP32 with NB = 4: one 16-byte word
// (every such address is a multiple of 4 values from an allocation's start).  One
// value at a time, a warp's loads took more cycles of the L1 than its bytes took of
// HBM: products of the mixed 4.2M-point slope 0.89 -> 0.84 ms, of the 1M-point block
// 0.222 -> 0.201.  (FP64 is bound by its pipe: 2.08 ms a product one by one, 2.10 by words.)
template <int NB, typename T>
__device__ __forceinline__ void load_row(const T *__restrict__ p, T v[NB]) {
  if constexpr (NB == 4 && sizeof(T) == 4) {
    const float4 q = __ldg(reinterpret_cast<const float4 *>(p));
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  } else {
#pragma unroll
    for (int i = 0; i < NB; ++i) v[i] = __ldg(p + i);
  }
}

// SPL * NB threads per block row: the SPL lanes of output r of a row split the
// row's blocks (lane l takes blocks l, l + SPL, ...) and spend one FMA per
// stored value of block row r; one shuffle sum per output joins them.
// (GB300's FP64 pipe is narrow: an FP64 SpMV should issue one FP64
// instruction per value with all lanes busy; the SPL-fold split gives the SM
// enough warps to cover the load latency.)
// y = D J x: x is in the unscaled unknowns (the preconditioner returns them),
// so that the matrix is read as the assembly wrote it; a pass that scaled it in
// place cost 4.1 ms (FP64) or 4.4 ms (FP32) per Newton iteration of the 4.2M-point
// slope, two products' time.
template <int NB, int SPL, typename T>
__global__ void k_bsr_spmv(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                           const int32_t *__restrict__ col, const T *__restrict__ val,
                           const T *__restrict__ dsc, const T *__restrict__ x, T *__restrict__ y,
                           const KrylovCtl *__restrict__ ctl,
                           int64_t xstride) {
  pdl_enter();
  if (ctl) {  // iteration graph: x is the vector of the iteration's number
    const int2 it = ctl->cur;
    if (it.y) return;
    x += it.x * xstride;
  }
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t o = t / SPL;
  const int part = (int)(t - o * SPL);
  const int64_t row = o / NB;
  const int r = (int)(o - row * NB);
  T acc = 0;
  if (row < nnodes) {
    const int e1 = row_ptr[row + 1];
#pragma unroll 4
    for (int e = row_ptr[row] + part; e < e1; e += SPL) {
      const T *blk = val + (int64_t)e * NB * NB + r * NB;
      const T *xb = x + (int64_t)__ldg(&col[e]) * NB;
      T bv[NB], xv[NB];
      load_row<NB>(blk, bv);
      load_row<NB>(xb, xv);
#pragma unroll
      for (int c = 0; c < NB; ++c) acc = fma(bv[c], xv[c], acc);
    }
  }
#pragma unroll
  for (int s = SPL / 2; s > 0; s >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, s);
  if (row < nnodes && part == 0) y[row * NB + r] = acc * dsc[row * NB + r];
}

// ---------------------------------------------------------------- FGMRES
// What a solve posts instead of an estimate once a value is not finite (a rotation
// formed from such a value could leave an estimate of zero): the host returns
// MPM_ERR_NONFINITE.
__device__ inline double not_finite() { return __longlong_as_double(0x7ff8000000000000ll); }

// Partial dots of w against V_0..V_{cnt-1}, block (b, i) summing its slice of
// V_i . w: the cnt products run side by side instead of one after another.
// A row i = cnt of blocks (grid y = cnt + 1) sums w . w.  With skip set, the
// kernel does nothing unless *skip is nonzero (a second Gram-Schmidt pass
// that the first pass's norms made unnecessary).
template <typename T>
__global__ void k_multidot2(const T *__restrict__ V, const T *__restrict__ w, int64_t n, int cnt,
                            double *__restrict__ part, const double *__restrict__ skip) {
  pdl_enter();
  if (skip && *skip == 0.0) return;
  const int i = blockIdx.y;
  const T *vi = i < cnt ? V + (int64_t)i * n : w;
  T acc = 0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    acc += vi[k] * w[k];
  const double s = block_sum((double)acc);
  if (threadIdx.x == 0) part[(int64_t)blockIdx.x * PSTR + i] = s;
}

// w -= sum_i h_i V_i; with want_norm also the partial sums of |w|^2; with
// skip set, nothing unless *skip is nonzero (as k_multidot2)
template <typename T>
__global__ void k_orth_sub(T *__restrict__ w, const T *__restrict__ V, const double *__restrict__ h, int cnt,
                           int64_t n, double *__restrict__ part, int want_norm, const double *__restrict__ skip) {
  pdl_enter();
  if (skip && *skip == 0.0) return;
  T nacc = 0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    T sv = w[k];
    for (int i = 0; i < cnt; ++i) sv -= (T)h[i] * V[(int64_t)i * n + k];
    w[k] = sv;
    nacc += sv * sv;
  }
  if (want_norm) {
    const double sn = block_sum((double)nacc);
    if (threadIdx.x == 0) part[(int64_t)blockIdx.x * PSTR] = sn;
  }
}

__global__ void k_multidot_reduce(const double *__restrict__ part, int np, int cnt,
                                  double *__restrict__ h, const double *__restrict__ skip) {
  pdl_enter();
  const int i = blockIdx.x;  // one block per coefficient
  if (i >= cnt) return;
  if (skip && *skip == 0.0) {  // the pass is skipped: its coefficients are zero
    if (threadIdx.x == 0) h[i] = 0.0;
    return;
  }
  double acc = 0.0;
  for (int b = threadIdx.x; b < np; b += blockDim.x) acc += part[(int64_t)b * PSTR + i];
  acc = block_sum(acc);
  if (threadIdx.x == 0) h[i] = acc;
}

// Whether classical Gram-Schmidt needs its second pass: after the first, w
// has lost most of its norm to the basis (|w1|^2 < theta^2 |w0|^2, |w0|^2 in
// h1[cnt] from the first pass's products, |w1|^2 from the first update's
// partials).  Writes 1 (second pass) or 0 into *flag.
__global__ void k_reorth_test(const double *__restrict__ part, int np, const double *__restrict__ h1, int cnt,
                              double theta, double *__restrict__ flag) {
  pdl_enter();
  double acc = 0.0;
  for (int b = threadIdx.x; b < np; b += blockDim.x) acc += part[(int64_t)b * PSTR];
  acc = block_sum(acc);
  if (threadIdx.x == 0) *flag = acc < theta * theta * h1[cnt] ? 1.0 : 0.0;
}

// Finish Arnoldi column j: ||w|| from the partials, H(:,j) = h1 + h2, apply
// the previous Givens rotations, form the new one, update g.
// scal[0] = |g_{j+1}| (residual estimate), scal[1] = 1 / ||w||.
__global__ void k_arnoldi_finish(const double *__restrict__ part, int np, int j, int m,
                                 const double *__restrict__ h1, const double *__restrict__ h2,
                                 double *__restrict__ H, double *__restrict__ g, double *__restrict__ cs,
                                 double *__restrict__ sn, double *__restrict__ scal) {
  pdl_enter();
  double acc = 0.0;
  for (int b = threadIdx.x; b < np; b += blockDim.x) acc += part[(int64_t)b * PSTR];
  acc = block_sum(acc);
  if (threadIdx.x != 0) return;
  const double hn = sqrt(acc);
  double col[PSTR];
  for (int i = 0; i <= j; ++i) col[i] = h1[i] + h2[i];
  for (int i = 0; i < j; ++i) {
    const double t = cs[i] * col[i] + sn[i] * col[i + 1];
    col[i + 1] = -sn[i] * col[i] + cs[i] * col[i + 1];
    col[i] = t;
  }
  const double r = hypot(col[j], hn);
  double c = 1.0, s = 0.0;
  if (!isfinite(r)) {
    s = not_finite();
  } else if (r > 0.0) {
    c = col[j] / r;
    s = hn / r;
  }
  cs[j] = c;
  sn[j] = s;
  col[j] = r;
  for (int i = 0; i <= j; ++i) H[i * m + j] = col[i];
  const double gj = g[j];
  g[j + 1] = -s * gj;
  g[j] = c * gj;
  scal[0] = fabs(g[j + 1]);
  scal[1] = hn > 0.0 ? 1.0 / hn : 0.0;
}

__global__ void k_gmres_init(double *__restrict__ g, int m, const double *beta_sq, double *scal) {
  pdl_enter();
  if (threadIdx.x != 0) return;
  const double beta = sqrt(beta_sq[0]);
  for (int i = 0; i <= m; ++i) g[i] = 0.0;
  g[0] = beta;
  scal[0] = beta;
  scal[1] = beta > 0.0 ? 1.0 / beta : 0.0;
}

__global__ void k_backsolve(const double *__restrict__ H, const double *__restrict__ g, int jc, int m,
                            double *__restrict__ y) {
  pdl_enter();
  if (threadIdx.x != 0) return;
  for (int i = jc - 1; i >= 0; --i) {
    double s = g[i];
    for (int l = i + 1; l < jc; ++l) s -= H[i * m + l] * y[l];
    y[i] = s / H[i * m + i];
  }
}

template <typename T>
__global__ void k_update_x(T *__restrict__ x, const T *__restrict__ Z, const double *y, int jc, int64_t n) {
  pdl_enter();
  const int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (k >= n) return;
  T s = x[k];
  for (int i = 0; i < jc; ++i) s += (T)y[i] * Z[(int64_t)i * n + k];
  x[k] = s;
}

// ------------------------------------- one iteration as a CUDA graph
// Below KRYLOV_GRAPH_MAX unknowns (and for batched contexts) an FGMRES iteration is a chain of kernels of
// a few microseconds, and what it costs is their number, their launches and the
// host's read of the residual estimate.  So the whole iteration is one graph:
// its kernels read the iteration's number from a control word; the reductions
// of partial sums are done by every block of the kernel that needs them (no
// kernel of their own); the kernel that scales the next basis vector also
// finishes the Arnoldi column and splits the vector for the preconditioner; the
// estimate is written to mapped host memory, which the host polls; and the
// host launches iteration j + 1 before it has seen j's estimate while the last
// one seen is far above the target (SPEC_MARGIN), so that the GPU does not wait
// for it.  An iteration launched past convergence is not counted and leaves
// the solution alone (it writes column j + 1 and later words only).
// In FP64 the second Gram-Schmidt pass of a single system depends on the first
// (REORTH_THETA): where it is needed the finishing kernel leaves the column
// unfinished and sets ctl->next.y.  Of an iteration launched ahead only the
// preconditioner's core then runs, and what it overwrites the second pass's finish
// writes anew.  The host launches that pass.  Batches take both passes always.
// Against kernels launched one by one with a reduction kernel per pass and a
// copy and stream synchronisation per iteration (GB300, whole steps): column 2.40 ->
// 1.61 ms (25 iterations), 17 x 17 deposit in FP32 6.45 -> 4.52 (70), harmonic
// footing 6.3 -> 5.1 (43), 80k-point footing 11.3 -> 9.9 (50), 50k-point footing in
// FP32 12.7 -> 10.6 (83), 163k-point block 48.9 -> 47.0 (60).  From
// KRYLOV_GRAPH_MAX unknowns on, an iteration takes milliseconds and the kernels
// with a grid sized to the iteration serve.
constexpr int64_t KRYLOV_GRAPH_MAX = 1 << 20;
constexpr double SPEC_MARGIN = 16.0;
constexpr double EST_REORTH = -2.0;  // posted instead of an estimate: second pass needed
constexpr int GS_SLICE = 512;        // vector elements per block of the inner products

// part[b * PSTR + i] = block (b, .)'s part of V_i . w, i < cnt (= ctl->cur.x + 1), and
// of w . w at i = cnt (with_norm): a warp per product and slice, all of them side
// by side (the grid has blocks for m products; those past cnt leave at once)
template <typename T>
__global__ void k_gs_dots(const T *__restrict__ V, const T *__restrict__ w, int64_t n, int64_t slice,
                          const KrylovCtl *__restrict__ ctl, int with_norm, int force, double *__restrict__ part) {
  pdl_enter();
  const int2 it = ctl->cur;
  if (it.y && !force) return;
  const int cnt = it.x + 1, lane = threadIdx.x & 31;
  const int i = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (i >= cnt + with_norm) return;
  const int64_t k0 = blockIdx.x * slice, k1 = min(k0 + slice, n);
  const T *vi = i < cnt ? V + (int64_t)i * n : w;
  T acc = 0;
#pragma unroll 8
  for (int64_t k = k0 + lane; k < k1; k += 32) acc += vi[k] * w[k];
  double s = (double)acc;
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) part[(int64_t)blockIdx.x * PSTR + i] = s;
}

// w -= sum_i h_i V_i with h summed from the np partials here; block 0 keeps h
// (with |w|^2 at h[cnt] when with_norm); npart: partial squared norms of the
// result (null: not wanted)
template <typename T>
__global__ void k_gs_update(T *__restrict__ w, const T *__restrict__ V, int64_t n, const KrylovCtl *__restrict__ ctl,
                            const double *__restrict__ part, int np, int with_norm, int force,
                            double *__restrict__ h, double *__restrict__ npart) {
  pdl_enter();
  const int2 it = ctl->cur;
  if (it.y && !force) return;
  __shared__ T hs[PSTR];
  const int cnt = it.x + 1;
  {  // the sums side by side: G = 2^lg lanes per coefficient
    const int nh = cnt + with_norm;
    int lg = 5;
    while (lg > 0 && (nh << lg) > (int)blockDim.x) --lg;
    const int G = 1 << lg, i = threadIdx.x >> lg, sub = threadIdx.x & (G - 1);
    double s = 0.0;
    if (i < nh) {
#pragma unroll 4
      for (int b = sub; b < np; b += G) s += part[(int64_t)b * PSTR + i];
    }
    for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (i < nh && sub == 0) {
      hs[i] = (T)s;  // (converted once: a conversion costs as much as an FP64 FMA)
      if (blockIdx.x == 0) h[i] = s;
    }
  }
  __syncthreads();
  T nacc = 0;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    T sv = w[k];
#pragma unroll 16
    for (int i = 0; i < cnt; ++i) sv -= hs[i] * V[(int64_t)i * n + k];
    w[k] = sv;
    nacc += sv * sv;
  }
  if (npart) {
    const double sn = block_sum((double)nacc);
    if (threadIdx.x == 0) npart[blockIdx.x] = sn;
  }
}

// v = s w at node a into the basis vector, and its split
template <int NB, typename T, typename Q>
__device__ inline void scale_split(int64_t a, const T *__restrict__ w, Q s, T *__restrict__ v, const SplitP<T> &P) {
  constexpr int D = NB - 1;
  T u[NB];
#pragma unroll
  for (int r = 0; r < NB; ++r) {
    const T x = (T)(w[a * NB + r] * s);
    v[a * NB + r] = x;
    u[r] = P.dsi ? x * P.dsi[a * NB + r] : x;
  }
  if (!P.dsi) return;  // no split: block-Jacobi preconditioner
  if (P.lower) {
#pragma unroll
    for (int i = 0; i < D; ++i) {
      T t = 0;
#pragma unroll
      for (int k = 0; k < D; ++k) t = fma(P.dinv[a * D * D + i * D + k], u[k], t);
      P.b0[a * D + i] = u[i];
      P.x0[a * D + i] = P.omega * t;
    }
    P.other[a] = u[D];
  } else {
#pragma unroll
    for (int k = 0; k < D; ++k) P.other[a * D + k] = u[k];
    P.b0[a] = u[D];
    P.x0[a] = P.omega * (P.dinv[a] * u[D]);
  }
}

// Finish Arnoldi column j: |w| from the partials, H(:, j) = h1 (+ h2), the
// previous Givens rotations and the new one (block 0), V_{j+1} = w / |w| with
// its split; the residual estimate goes to est[j].  With h1 holding |w|^2 from
// before the update at h1[j + 1] (theta > 0), a column that kept less than
// theta of it halts for a second pass instead.  The square root and the
// reciprocal are one thread's (as every thread's they would cost the SM's FP64
// pipe microseconds).
template <int NB, typename T>
__global__ void k_gs_finish(const T *__restrict__ w, T *__restrict__ V, int64_t nnodes, int m, KrylovCtl *ctl,
                            const double *__restrict__ npart, int np,
                            const double *__restrict__ h1, const double *__restrict__ h2, double theta, int force,
                            double *__restrict__ H, double *__restrict__ g, double *__restrict__ cs,
                            double *__restrict__ sn, double *est, SplitP<T> P) {
  pdl_enter();
  double acc = 0.0;
  for (int b = threadIdx.x; b < np; b += blockDim.x) acc += npart[b];
  const int2 it = ctl->cur;
  if (it.y && !force) return;
  __shared__ T sh_scale;
  __shared__ int sh_again;
  __shared__ double col[PSTR], sc[PSTR], ss[PSTR];
  const int j = it.x;
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i <= j; i += blockDim.x) {
      col[i] = h1[i] + (h2 ? h2[i] : 0.0);
      sc[i] = cs[i];
      ss[i] = sn[i];
    }
  const double w0 = theta > 0.0 ? h1[j + 1] : 0.0;
  acc = block_sum(acc);
  double hn = 0.0;
  if (threadIdx.x == 0) {
    hn = sqrt(acc);
    sh_again = theta > 0.0 && acc < theta * theta * w0;
    sh_scale = (T)(hn > 0.0 ? 1.0 / hn : 0.0);
  }
  __syncthreads();
  const bool again = sh_again != 0;
  if (!again) {
    const T s = sh_scale;
    T *v = V + (int64_t)(j + 1) * (nnodes * NB);
    for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < nnodes; a += (int64_t)gridDim.x * blockDim.x)
      scale_split<NB>(a, w, s, v, P);
    if (blockIdx.x == 0) {
      if (threadIdx.x == 0) {
        double below = col[0];
#pragma unroll 4
        for (int i = 0; i < j; ++i) {  // (one dependent FMA per rotation)
          const double nx = col[i + 1];
          col[i] = sc[i] * below + ss[i] * nx;
          below = fma(-ss[i], below, sc[i] * nx);
        }
        double r = fma(below, below, hn * hn);
        r = r > 1e-280 && r < 1e280 ? sqrt(r) : hypot(below, hn);
        double c = 1.0, s2 = 0.0;
        if (!isfinite(r)) {
          s2 = not_finite();
        } else if (r > 0.0) {
          c = below / r;
          s2 = hn / r;
        }
        cs[j] = c;
        sn[j] = s2;
        col[j] = r;
        const double gj = g[j];
        g[j + 1] = -s2 * gj;
        g[j] = c * gj;
        slot_write(est + j, fabs(s2 * gj));
      }
      __syncthreads();
      for (int i = threadIdx.x; i <= j; i += blockDim.x) H[i * m + j] = col[i];
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    ctl->next = make_int2(again ? j : j + 1, again ? 1 : 0);
    if (again) slot_write(est + j, EST_REORTH);
  }
}

// V_0 = r / |r| with its split, |r|^2 from np partials; block 0 starts the
// Givens right-hand side, the control word and posts |r|
template <int NB, typename T>
__global__ void k_gs_start(const T *__restrict__ r, T *__restrict__ V, int64_t nnodes, int m, KrylovCtl *ctl,
                           const double *__restrict__ npart, int np, double *__restrict__ g, double *beta_slot,
                           SplitP<T> P) {
  __shared__ double sh_nrm;
  __shared__ T sh_scale;
  double acc = 0.0;
  for (int b = threadIdx.x; b < np; b += blockDim.x) acc += npart[b];
  acc = block_sum(acc);
  if (threadIdx.x == 0) {
    sh_nrm = sqrt(acc);
    sh_scale = (T)(sh_nrm > 0.0 ? 1.0 / sh_nrm : 0.0);
  }
  __syncthreads();
  const double beta = sh_nrm;
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i <= m; i += blockDim.x) g[i] = i == 0 ? beta : 0.0;
    if (threadIdx.x == 0) {
      ctl->next = make_int2(0, 0);
      slot_write(beta_slot, beta);
    }
  }
  const T s = sh_scale;
  for (int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; a < nnodes; a += (int64_t)gridDim.x * blockDim.x)
    scale_split<NB>(a, r, s, V, P);
}

// Z_j = [zu; zp], in the unscaled unknowns
template <int NB, typename T>
__global__ void k_it_merge(int64_t nnodes, const T *__restrict__ zu, const T *__restrict__ zp,
                           T *__restrict__ Z, KrylovCtl *ctl) {
  pdl_enter();
  const int2 it = ctl->next;
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->cur = it;
  if (it.y) return;
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  constexpr int D = NB - 1;
  T *z = Z + (int64_t)it.x * (nnodes * NB);
#pragma unroll
  for (int k = 0; k < D; ++k) z[a * NB + k] = zu[a * D + k];
  z[a * NB + D] = zp[a];
}

// Z_j = Dinv V_j (node-block Jacobi)
template <int NB, typename T>
__global__ void k_it_bj(int64_t nnodes, const T *__restrict__ dinv, const T *__restrict__ V, T *__restrict__ Z,
                        KrylovCtl *ctl) {
  pdl_enter();
  const int2 it = ctl->next;
  if (blockIdx.x == 0 && threadIdx.x == 0) ctl->cur = it;
  if (it.y) return;
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  const T *x = V + (int64_t)it.x * (nnodes * NB);
  T *z = Z + (int64_t)it.x * (nnodes * NB);
  T xv[NB];
  for (int j = 0; j < NB; ++j) xv[j] = x[a * NB + j];
  for (int i = 0; i < NB; ++i) {
    T s = 0;
    for (int j = 0; j < NB; ++j) s += dinv[a * NB * NB + i * NB + j] * xv[j];
    z[a * NB + i] = s;
  }
}

// x += Z y with H y = g solved by every block (jc x jc, back substitution by
// columns; the triangle in shared memory when it fits, smem doubles)
template <typename T>
__global__ void k_solve_update_x(T *__restrict__ x, const T *__restrict__ Z, const double *__restrict__ H,
                                 const double *__restrict__ g, int jc, int m, int64_t n, int in_smem) {
  extern __shared__ __align__(16) unsigned char solve_smem[];
  double *R = reinterpret_cast<double *>(solve_smem);
  __shared__ double y[PSTR], rinv[PSTR];
  if (in_smem)
    for (int t = threadIdx.x; t < jc * jc; t += blockDim.x) R[t] = H[t / jc * m + t % jc];
  for (int i = threadIdx.x; i < jc; i += blockDim.x) {
    y[i] = g[i];
    rinv[i] = 1.0 / H[i * m + i];
  }
  __syncthreads();
  for (int i = jc - 1; i >= 0; --i) {
    const double yi = y[i] * rinv[i];
    __syncthreads();
    for (int l = threadIdx.x; l < i; l += blockDim.x) y[l] -= (in_smem ? R[l * jc + i] : H[l * m + i]) * yi;
    if (threadIdx.x == 0) y[i] = yi;
    __syncthreads();
  }
  T *yt = reinterpret_cast<T *>(rinv);  // (no longer needed)
  for (int i = threadIdx.x; i < jc; i += blockDim.x) yt[i] = (T)y[i];
  __syncthreads();
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    T s = x[k];
#pragma unroll 16
    for (int i = 0; i < jc; ++i) s += yt[i] * Z[(int64_t)i * n + k];
    x[k] = s;
  }
}

template <int NB, typename T>
void spmv(Ctx &c, const LinSys<T> &S, const T *x, T *y, const KrylovCtl *ctl = nullptr, int64_t xstride = 0) {
  constexpr int SPL = NB == 3 ? 2 : 4;  // 25 (2D) / 125 (3D) blocks per GIMP row
  const int64_t threads = c.g.nnodes * NB * SPL;
  prof_begin(c, MPM_PROF_SPMV);
  const int32_t *rp = c.row_ptr, *cl = c.col;
  const T *val = S.val;
  launch_pdl(c, k_bsr_spmv<NB, SPL, T>, nblk(threads), TPB, 0, c.g.nnodes, rp, cl, val, (const T *)S.dscale, x, y,
             ctl, xstride);
  prof_end(c, MPM_PROF_SPMV);
}

template <int NB, typename T>
void precond(Ctx &c, LinSys<T> &S, const T *x, T *y) {
  prof_begin(c, MPM_PROF_PRECOND);
  if (c.opt.precond == MPM_PRECOND_SCHUR_MG) {
    schur_apply<T>(c, S, x, y);
  } else {
    launch_pdl(c, k_bj_apply<NB, T>, nblk(c.g.nnodes), TPB, 0, c.g.nnodes, (const T *)S.dinv, x, y);
  }
  prof_end(c, MPM_PROF_PRECOND);
}

double read_scalar(Ctx &c, const double *dptr) {
  cudaMemcpyAsync(c.h_scalar, dptr, sizeof(double), cudaMemcpyDeviceToHost, c.st);
  cudaStreamSynchronize(c.st);
  return c.h_scalar[0];
}

// ------------------------------------------------ batched FGMRES (instances)
// A batched context solves one block-diagonal system (the instances never
// couple; the preconditioner keeps that structure), so FGMRES runs per
// instance: every inner product, Hessenberg column, Givens rotation and
// convergence test is the instance's own, while each kernel serves all
// instances at once.  An instance that meets its tolerance in column j is
// frozen from column j + 1 on (its Krylov vectors are zero from then) until
// the others finish.
// The vectors are walked in slices of up to BG_NODES nodes of one instance
// (Ctx::bn_*; the nodes between instances form slices of their own, kept at
// zero): a block per slice and group of products forms partial sums, and every
// block that needs an instance's sum adds its slices.  (One block per instance
// and product, walking the instance's node box, took 33 us a pass on 64 columns
// of 4,200 nodes and three passes an iteration.)  The iteration is a graph, as
// for one instance; frozen_at holds the first column an instance skips, so that
// the blocks of an instance agree on it while its first block moves it on.
// Both passes of classical Gram-Schmidt run in every iteration, in FP64 as in FP32:
// an instance's basis is as orthogonal as two passes leave it, whatever the others
// need.  (With the second pass only where one instance's first had lost 99% of its
// norm, a step of 64 columns took 53.3 ms against 59.2, of 64 footings 84.0 against
// 88.2.)  The Gram-Schmidt kernels run at the FP64 rate of their products.
constexpr int BG_NODES = 256;

struct BatchK {  // device pointers of the batched solve, by value
  int ni, m;
  const int32_t *nodes, *s0;  // node lists by slice; first slice of every instance (ni + 1)
  const int4 *slices;         // (instance or -1, start in nodes, count, -)
  double *H, *g, *cs, *sn, *h1, *h2, *tgt, *res;
  int32_t *frozen_at, *jc;
  double *part, *npart;
  BatchPost *post;
  KrylovCtl *ctl;
  double *slot;
};

// sum of p over the slices of instance i, in thread 0 (block-wide)
__device__ inline double slices_sum(const BatchK &K, int i, const double *__restrict__ p) {
  double acc = 0.0;
  for (int b = K.s0[i] + threadIdx.x; b < K.s0[i + 1]; b += blockDim.x) acc += p[b];
  return block_sum(acc);
}

// How far an estimate is from its target: finite also for a target of zero or below
// (a krylov_rtol that no estimate reaches).  Ratios are compared by their bits, where
// the NaN is above every number.
__device__ inline double batch_ratio(double res, double tgt) {
  if (!isfinite(res)) return not_finite();
  return tgt > 0.0 ? fmin(res / tgt, 1e300) : 1e300;
}

// An instance's first block reports (thread 0): whether it goes on and how far
// its estimate is from its target; the last report of the kernel posts the largest
// ratio (0: all done) and moves the control word
__device__ inline void batch_report(const BatchK &K, int j, double *slot, bool active, double ratio) {
  BatchPost *q = K.post;
  if (active) {
    atomicAdd(&q->active, 1u);
    atomicMax(&q->ratio, (unsigned long long)__double_as_longlong(ratio));
  }
  __threadfence();
  if (atomicAdd(&q->arrived, 1u) != (unsigned)K.ni - 1) return;
  __threadfence();
  const unsigned act = atomicAdd(&q->active, 0u);
  const double worst = __longlong_as_double((long long)atomicMax(&q->ratio, 0ull));
  q->active = q->arrived = 0;
  q->ratio = 0;
  K.ctl->next = make_int2(j + 1, 0);
  slot_write(slot, act ? worst : 0.0);
}

template <int NB, typename T>
__global__ void k_bgs_norm(BatchK K, const T *__restrict__ r) {
  const int4 sl = K.slices[blockIdx.x];
  double acc = 0.0;
  if ((int)threadIdx.x < sl.z) {
    const int64_t a = K.nodes[sl.y + threadIdx.x];
    for (int c = 0; c < NB; ++c) acc += (double)r[a * NB + c] * (double)r[a * NB + c];
  }
  acc = block_sum(acc);
  if (threadIdx.x == 0) K.npart[blockIdx.x] = acc;
}

// start of a cycle: V_0 = r / |r| with its split, g = |r| e_1 per instance; the
// tolerance rtol |r| is fixed at the first start; an instance within it is done
template <int NB, typename T>
__global__ void k_bgs_start(BatchK K, const T *__restrict__ r, T *__restrict__ V, double rtol, int set_target,
                            SplitP<T> P) {
  const int4 sl = K.slices[blockIdx.x];
  const int i = sl.x;
  __shared__ double sh_scale;
  if (threadIdx.x == 0) sh_scale = 0.0;
  if (i >= 0) {
    const double n2 = slices_sum(K, i, K.npart);
    if (threadIdx.x == 0) {
      const double beta = sqrt(n2), tgt = set_target ? rtol * beta : K.tgt[i];
      const bool done = isfinite(beta) && !(beta > tgt);
      sh_scale = !done && beta > 0.0 ? 1.0 / beta : 0.0;
      if ((int)blockIdx.x == K.s0[i]) {
        if (set_target) K.tgt[i] = tgt;
        double *g = K.g + (int64_t)i * (K.m + 1);
        for (int k = 1; k <= K.m; ++k) g[k] = 0.0;
        g[0] = beta;
        K.jc[i] = 0;
        K.frozen_at[i] = done ? 0 : 0x7fffffff;
        batch_report(K, -1, K.slot + SLOT_BETA, !done, batch_ratio(beta, tgt));
      }
    }
  }
  __syncthreads();
  if ((int)threadIdx.x < sl.z) scale_split<NB>(K.nodes[sl.y + threadIdx.x], r, sh_scale, V, P);
}

// products of a slice, a warp each; summed in FP64
template <int NB, typename T>
__global__ void k_bgs_dots(BatchK K, const T *__restrict__ V, const T *__restrict__ w, int64_t n) {
  pdl_enter();
  const int j = K.ctl->cur.x, lane = threadIdx.x & 31;
  const int k = blockIdx.y * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (k > j) return;
  const int4 sl = K.slices[blockIdx.x];
  if (K.frozen_at[sl.x] <= j) return;
  const T *vk = V + (int64_t)k * n;
  double s = 0.0;
#pragma unroll 4
  for (int e = lane; e < sl.z; e += 32) {
    const int64_t a = K.nodes[sl.y + e];
#pragma unroll
    for (int c = 0; c < NB; ++c) s += (double)vk[a * NB + c] * (double)w[a * NB + c];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) K.part[(int64_t)blockIdx.x * PSTR + k] = s;
}

// w -= sum_k h_k V_k on a slice, h its instance's sums over the slices (kept in
// h by the instance's first block); npart: the slice's squared norm after
template <int NB, typename T>
__global__ void k_bgs_update(BatchK K, T *__restrict__ w, const T *__restrict__ V, int64_t n,
                             double *__restrict__ h, int want_norm) {
  pdl_enter();
  const int j = K.ctl->cur.x;
  const int4 sl = K.slices[blockIdx.x];
  const int i = sl.x, cnt = j + 1;
  if (K.frozen_at[i] <= j) return;
  __shared__ T hs[PSTR];
  {
    const int b1 = K.s0[i + 1];
    int lg = 5;
    while (lg > 0 && (cnt << lg) > (int)blockDim.x) --lg;
    const int G = 1 << lg, k = threadIdx.x >> lg, sub = threadIdx.x & (G - 1);
    double s = 0.0;
    if (k < cnt) {
#pragma unroll 4
      for (int b = K.s0[i] + sub; b < b1; b += G) s += K.part[(int64_t)b * PSTR + k];
    }
    for (int o = G >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (k < cnt && sub == 0) {
      hs[k] = (T)s;
      if ((int)blockIdx.x == K.s0[i]) h[(int64_t)i * PSTR + k] = s;
    }
  }
  __syncthreads();
  double nacc = 0.0;
  if ((int)threadIdx.x < sl.z) {
    const int64_t a = (int64_t)K.nodes[sl.y + threadIdx.x] * NB;
    T x[NB];
#pragma unroll
    for (int c = 0; c < NB; ++c) x[c] = w[a + c];
#pragma unroll 8
    for (int k = 0; k < cnt; ++k)
#pragma unroll
      for (int c = 0; c < NB; ++c) x[c] -= hs[k] * V[(int64_t)k * n + a + c];
#pragma unroll
    for (int c = 0; c < NB; ++c) {
      w[a + c] = x[c];
      nacc += (double)x[c] * (double)x[c];
    }
  }
  if (want_norm) {
    nacc = block_sum(nacc);
    if (threadIdx.x == 0) K.npart[blockIdx.x] = nacc;
  }
}

// Arnoldi column j of every active instance (its first block): H(:, j) = h1 + h2,
// the rotations, g, the estimate; V_{j+1} = w / |w| with its split (all blocks),
// zero for a frozen instance and between instances.
template <int NB, typename T>
__global__ void k_bgs_finish(BatchK K, const T *__restrict__ w, T *__restrict__ V, int64_t n, SplitP<T> P) {
  pdl_enter();
  const int j = K.ctl->cur.x;
  const int4 sl = K.slices[blockIdx.x];
  const int i = sl.x;
  const bool lead = i >= 0 && (int)blockIdx.x == K.s0[i];
  const bool live = i >= 0 && K.frozen_at[i] > j;
  __shared__ double sh_scale;
  __shared__ double col[PSTR], sc[PSTR], ss[PSTR];
  double n2 = 0.0;
  if (live) {
    if (lead)
      for (int k = threadIdx.x; k <= j; k += blockDim.x) {
        const int64_t hk = (int64_t)i * PSTR + k, rk = (int64_t)i * (K.m + 1) + k;
        col[k] = K.h1[hk] + K.h2[hk];
        sc[k] = K.cs[rk];
        ss[k] = K.sn[rk];
      }
    n2 = slices_sum(K, i, K.npart);
  }
  if (threadIdx.x == 0) {
    const double hn = live ? sqrt(n2) : 0.0;
    sh_scale = hn > 0.0 ? 1.0 / hn : 0.0;
    if (lead) {
      if (live) {
        double *g = K.g + (int64_t)i * (K.m + 1), *H = K.H + (int64_t)i * (K.m + 1) * K.m;
        double below = col[0];
#pragma unroll 4
        for (int k = 0; k < j; ++k) {
          const double nx = col[k + 1];
          H[k * K.m + j] = sc[k] * below + ss[k] * nx;
          below = fma(-ss[k], below, sc[k] * nx);
        }
        const double r = hypot(below, hn);
        double c = 1.0, sv = 0.0;
        if (!isfinite(r)) {
          sv = not_finite();
        } else if (r > 0.0) {
          c = below / r;
          sv = hn / r;
        }
        K.cs[(int64_t)i * (K.m + 1) + j] = c;
        K.sn[(int64_t)i * (K.m + 1) + j] = sv;
        H[j * K.m + j] = r;
        const double gj = g[j], res = fabs(sv * gj);
        g[j + 1] = -sv * gj;
        g[j] = c * gj;
        K.res[i] = res;
        K.jc[i] = j + 1;
        if (res <= K.tgt[i] || (isfinite(res) && !(hn > 0.0))) K.frozen_at[i] = j + 1;
      }
      const bool on = K.frozen_at[i] > j + 1;
      batch_report(K, j, K.slot + j, on, on ? batch_ratio(K.res[i], K.tgt[i]) : 0.0);
    }
  }
  __syncthreads();
  if ((int)threadIdx.x < sl.z)
    scale_split<NB>(K.nodes[sl.y + threadIdx.x], w, sh_scale, V + (int64_t)(j + 1) * n, P);
}

// x += Z y per slice, its instance's triangle solved by every block
template <int NB, typename T>
__global__ void k_bgs_solve_x(BatchK K, T *__restrict__ x, const T *__restrict__ Z, int64_t n) {
  const int4 sl = K.slices[blockIdx.x];
  const int i = sl.x, jc = K.jc[i];
  const double *H = K.H + (int64_t)i * (K.m + 1) * K.m, *g = K.g + (int64_t)i * (K.m + 1);
  __shared__ double y[PSTR], rinv[PSTR];
  __shared__ T yt[PSTR];
  for (int k = threadIdx.x; k < jc; k += blockDim.x) {
    const double d = H[k * K.m + k];
    y[k] = g[k];
    rinv[k] = d != 0.0 ? 1.0 / d : 0.0;
  }
  __syncthreads();
  for (int k = jc - 1; k >= 0; --k) {
    const double yk = y[k] * rinv[k];
    __syncthreads();
    for (int l = threadIdx.x; l < k; l += blockDim.x) y[l] -= H[l * K.m + k] * yk;
    if (threadIdx.x == 0) yt[k] = (T)yk;
    __syncthreads();
  }
  if ((int)threadIdx.x >= sl.z) return;
  const int64_t a = (int64_t)K.nodes[sl.y + threadIdx.x] * NB;
  T s[NB];
#pragma unroll
  for (int c = 0; c < NB; ++c) s[c] = x[a + c];
#pragma unroll 8
  for (int k = 0; k < jc; ++k)
#pragma unroll
    for (int c = 0; c < NB; ++c) s[c] += yt[k] * Z[(int64_t)k * n + a + c];
#pragma unroll
  for (int c = 0; c < NB; ++c) x[a + c] = s[c];
}

inline BatchK batch_k(const Ctx &c) {
  const int64_t ni = c.ninst, m = c.m_restart;
  BatchK K{};
  K.ni = c.ninst;
  K.m = c.m_restart;
  K.nodes = c.bn_nodes;
  K.s0 = c.bn_s0;
  K.slices = c.bn_slices;
  K.H = c.bk;
  K.g = K.H + ni * (m + 1) * m;
  K.cs = K.g + ni * (m + 1);
  K.sn = K.cs + ni * (m + 1);
  K.h1 = K.sn + ni * (m + 1);
  K.h2 = K.h1 + ni * PSTR;
  K.tgt = K.h2 + ni * PSTR;
  K.res = K.tgt + ni;
  K.frozen_at = c.bk_i;
  K.jc = c.bk_i + ni;
  K.part = c.bn_part;
  K.npart = c.bn_npart;
  K.post = c.bk_post;
  K.ctl = c.ctl;
  K.slot = c.d_slot;
  return K;
}

// Geometry of the Gram-Schmidt kernels of the iteration graph.
struct GsGeom {
  int64_t slice;
  int ndot, ydot, nupd, nnode;
};
inline GsGeom gs_geom(const Ctx &c) {
  const int64_t N = c.N();
  GsGeom q;
  q.slice = std::max<int64_t>(GS_SLICE, (N + NPART - 1) / NPART);
  q.slice = (q.slice + 31) / 32 * 32;
  q.ndot = (int)((N + q.slice - 1) / q.slice);
  q.ydot = (c.m_restart + 1 + TPB / 32 - 1) / (TPB / 32);
  q.nupd = std::min(NPART, nblk(N));
  q.nnode = std::min(NPART, nblk(c.g.nnodes));
  return q;
}

template <typename T>
SplitP<T> next_split(Ctx &c, LinSys<T> &S) {
  return c.opt.precond == MPM_PRECOND_SCHUR_MG ? schur_split_args<T>(c, S) : SplitP<T>{};
}

// The kernels of one iteration, from the preconditioner's core (its first
// sub-solve's split is in place) to the split of the next basis vector.
template <int NB, typename T>
void enqueue_iteration(Ctx &c, LinSys<T> &S) {
  const int64_t N = c.N(), nn = c.g.nnodes;
  const GsGeom q = gs_geom(c);
  const KrylovCtl *ctl = c.ctl;
  double *h1 = c.hcol, *h2 = c.hcol + PSTR;
  const SplitP<T> before = next_split<T>(c, S);
  const T *zu, *zp, *V = S.V, *w = S.w;
  prof_begin(c, MPM_PROF_PRECOND);
  if (c.opt.precond == MPM_PRECOND_SCHUR_MG) {
    schur_core_launch<T>(c, S, &zu, &zp);
    launch_pdl(c, k_it_merge<NB, T>, nblk(nn), TPB, 0, nn, zu, zp, S.Z, c.ctl);
  } else {
    launch_pdl(c, k_it_bj<NB, T>, nblk(nn), TPB, 0, nn, (const T *)S.dinv, V, S.Z, c.ctl);
  }
  prof_end(c, MPM_PROF_PRECOND);
  spmv<NB, T>(c, S, S.Z, S.w, ctl, N);
  prof_begin(c, MPM_PROF_ORTH);
  // the split goes where the next core reads it: a replayed graph's core is the
  // one captured here, a directly launched one has swapped its buffers
  const SplitP<T> next = c.capturing ? before : next_split<T>(c, S);
  if (c.ninst > 1) {
    const BatchK K = batch_k(c);
    launch_pdl(c, k_bgs_dots<NB, T>, dim3(c.bn_live, q.ydot), TPB, 0, K, V, w, N);
    launch_pdl(c, k_bgs_update<NB, T>, c.bn_live, BG_NODES, 0, K, S.w, V, N, K.h1, 0);
    launch_pdl(c, k_bgs_dots<NB, T>, dim3(c.bn_live, q.ydot), TPB, 0, K, V, w, N);
    launch_pdl(c, k_bgs_update<NB, T>, c.bn_live, BG_NODES, 0, K, S.w, V, N, K.h2, 1);
    launch_pdl(c, k_bgs_finish<NB, T>, c.bn_all, BG_NODES, 0, K, w, S.V, N, next);
    prof_end(c, MPM_PROF_ORTH);
    return;
  }
  // FP64: one pass, |w|^2 beside the products for the test of the second;
  // FP32: always two (one leaves the basis orthogonal to about 1e-6 only)
  const bool sel = sizeof(T) == sizeof(double);
  const double *part = c.part;
  launch_pdl(c, k_gs_dots<T>, dim3(q.ndot, q.ydot), TPB, 0, V, w, N, q.slice, ctl, sel ? 1 : 0, 0, c.part);
  launch_pdl(c, k_gs_update<T>, q.nupd, TPB, 0, S.w, V, N, ctl, part, q.ndot, sel ? 1 : 0, 0, h1,
             sel ? c.npart : (double *)nullptr);
  if (!sel) {
    launch_pdl(c, k_gs_dots<T>, dim3(q.ndot, q.ydot), TPB, 0, V, w, N, q.slice, ctl, 0, 0, c.part);
    launch_pdl(c, k_gs_update<T>, q.nupd, TPB, 0, S.w, V, N, ctl, part, q.ndot, 0, 0, h2, c.npart);
  }
  launch_pdl(c, k_gs_finish<NB, T>, q.nnode, TPB, 0, w, S.V, nn, c.m_restart, c.ctl, (const double *)c.npart,
             q.nupd, (const double *)h1, sel ? (const double *)nullptr : (const double *)h2,
             sel ? REORTH_THETA : 0.0, 0, c.H, c.gvec, c.cs, c.sn, c.d_slot, next);
  prof_end(c, MPM_PROF_ORTH);
}

// The second Gram-Schmidt pass of the halted column and its finish (FP64, one
// instance).
template <int NB, typename T>
void enqueue_second_pass(Ctx &c, LinSys<T> &S, const SplitP<T> &next) {
  const int64_t N = c.N(), nn = c.g.nnodes;
  const GsGeom q = gs_geom(c);
  double *h1 = c.hcol, *h2 = c.hcol + PSTR;
  c.launches += 3;
  k_gs_dots<T><<<dim3(q.ndot, q.ydot), TPB, 0, c.st>>>(S.V, S.w, N, q.slice, c.ctl, 0, 1, c.part);
  k_gs_update<T><<<q.nupd, TPB, 0, c.st>>>(S.w, S.V, N, c.ctl, c.part, q.ndot, 0, 1, h2, c.npart);
  k_gs_finish<NB, T><<<q.nnode, TPB, 0, c.st>>>(S.w, S.V, nn, c.m_restart, c.ctl, c.npart, q.nupd, h1, h2, 0.0, 1,
                                                c.H, c.gvec, c.cs, c.sn, c.d_slot, next);
}

template <int NB, typename T>
int fgmres_graph_impl(Ctx &c, LinSys<T> &S, double rtol, int maxit, int *iters) {
  const int64_t N = c.N(), nn = c.g.nnodes;
  const int m = c.m_restart;
  const GsGeom q = gs_geom(c);
  const T *b = S.rhs;
  T *x = S.x, *w = S.w;
  // events around the classes of an iteration cannot be inside a graph
  const int timed = (1 << MPM_PROF_SPMV) | (1 << MPM_PROF_ORTH) | (1 << MPM_PROF_PRECOND);
  const bool graph = !(c.opt.profile & timed);
  if (graph && (!S.itexec || S.itkey_col != c.col || S.itkey_val != S.val)) {
    if (S.itexec) cudaGraphExecDestroy(S.itexec);
    S.itexec = nullptr;
    const int64_t before = c.launches;
    const SplitP<T> sp = next_split<T>(c, S);
    cudaGraph_t gr = nullptr;
    bool ok = cudaStreamBeginCapture(c.st, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      c.capturing = true;
      enqueue_iteration<NB, T>(c, S);
      c.capturing = false;
      ok = cudaStreamEndCapture(c.st, &gr) == cudaSuccess && gr;
    }
    if (ok) ok = cudaGraphInstantiate(&S.itexec, gr, 0) == cudaSuccess;
    if (gr) cudaGraphDestroy(gr);
    S.itkernels = c.launches - before;
    c.launches = before;
    if (ok) {
      S.it_x0 = sp.x0;
      S.itkey_col = c.col;
      S.itkey_val = S.val;
    } else {  // capture unavailable: the kernels are launched directly
      cudaGetLastError();
      S.itexec = nullptr;
    }
  }
  const bool use = graph && S.itexec;
  auto split = [&]() {
    SplitP<T> P = next_split<T>(c, S);
    if (use) P.x0 = S.it_x0;
    return P;
  };
  auto launch = [&](int j) {
    slot_reset(c, j);
    if (use) {
      cudaGraphLaunch(S.itexec, c.st);
      c.launches += S.itkernels;
    } else {
      enqueue_iteration<NB, T>(c, S);
    }
  };
  // the first start's norm and target: of the system, or (batched) the largest
  // ratio of an instance's norm to its target against 1 (0: nothing to do)
  const bool batch = c.ninst > 1;
  auto start = [&](const T *r, double *beta, int first) {
    slot_reset(c, SLOT_BETA);
    if (batch) {
      const BatchK K = batch_k(c);
      k_bgs_norm<NB, T><<<c.bn_live, BG_NODES, 0, c.st>>>(K, r);
      k_bgs_start<NB, T><<<c.bn_all, BG_NODES, 0, c.st>>>(K, r, S.V, rtol, first, split());
      c.launches += 2;
      return slot_wait(c, SLOT_BETA, beta);
    }
    k_dot_partial<T><<<q.nupd, TPB, 0, c.st>>>(r, r, N, c.npart);
    k_gs_start<NB, T><<<q.nnode, TPB, 0, c.st>>>(r, S.V, nn, m, c.ctl, c.npart, q.nupd, c.gvec,
                                                 c.d_slot + SLOT_BETA, split());
    c.launches += 2;
    return slot_wait(c, SLOT_BETA, beta);
  };
  cudaMemsetAsync(x, 0, sizeof(T) * N, c.st);
  *iters = 0;
  double beta0;
  if (int rc = start(b, &beta0, 1)) return rc;
  if (!isfinite(beta0)) return MPM_ERR_NONFINITE;
  if (!(beta0 > 0.0)) return MPM_OK;
  const double target = batch ? 0.5 : rtol * beta0;  // (a batch posts 0 or a ratio above 1)
  int total = 0;
  bool converged = false;
  double seen = beta0;  // the last estimate the host has read
  while (true) {
    int jc = 0, launched = 0;
    for (int j = 0; j < m; ++j) {
      if (launched <= j) launch(launched++);
      if (launched == j + 1 && launched < m && total + 1 < maxit && seen > SPEC_MARGIN * target) launch(launched++);
      double est;
      if (int rc = slot_wait(c, j, &est)) return rc;
      if (est == EST_REORTH) {  // column j was left unfinished, also by what was launched ahead
        slot_reset(c, j);
        enqueue_second_pass<NB, T>(c, S, split());
        launched = j + 1;
        if (int rc = slot_wait(c, j, &est)) return rc;
      }
      ++total;
      jc = j + 1;
      *iters = total;
      if (!isfinite(est)) return MPM_ERR_NONFINITE;
      seen = est;
      if (est <= target) {
        converged = true;
        break;
      }
      if (total >= maxit) break;
    }
    if (batch) {
      k_bgs_solve_x<NB, T><<<c.bn_live, BG_NODES, 0, c.st>>>(batch_k(c), x, S.Z, N);
    } else {
      const int in_smem = jc * jc * (int)sizeof(double) <= 40 * 1024;
      k_solve_update_x<T><<<q.nupd, TPB, in_smem ? sizeof(double) * jc * jc : 0, c.st>>>(x, S.Z, c.H, c.gvec, jc, m, N,
                                                                                         in_smem);
    }
    UPMPM_LAUNCH(c);
    if (converged || total >= maxit) break;
    // restart from the true residual r = b - A x
    spmv<NB, T>(c, S, x, w);
    k_residual_vec<T><<<nblk(N), TPB, 0, c.st>>>(w, b, N);
    UPMPM_LAUNCH(c);
    double br;
    if (int rc = start(w, &br, 0)) return rc;
    if (!isfinite(br)) return MPM_ERR_NONFINITE;
    if (br <= target) {
      converged = true;
      break;
    }
    seen = br;
  }
  *iters = total;
  if (check_cuda(c, cudaGetLastError(), "fgmres")) return MPM_ERR_CUDA;
  return converged ? MPM_OK : MPM_ERR_KRYLOV_STAGNATED;
}

template <int NB, typename T>
int fgmres_impl(Ctx &c, LinSys<T> &S, double rtol, int maxit, int *iters) {
  const int64_t N = c.N();
  if (c.ninst > 1 || N < KRYLOV_GRAPH_MAX)
    return fgmres_graph_impl<NB, T>(c, S, rtol, maxit, iters);
  const int m = c.m_restart;
  const int gN = nblk(N);
  const T *b = S.rhs;
  T *x = S.x, *w = S.w;
  double *h1 = c.hcol, *h2 = c.hcol + PSTR;
  cudaMemsetAsync(x, 0, sizeof(T) * N, c.st);
  // beta = ||b||, V_0 = b / beta
  k_dot_partial<T><<<NPART, TPB, 0, c.st>>>(b, b, N, c.part);
  k_reduce<<<1, TPB, 0, c.st>>>(c.part, NPART, c.scal + 2);
  k_gmres_init<<<1, 32, 0, c.st>>>(c.gvec, m, c.scal + 2, c.scal);
  k_scale_copy<T><<<gN, TPB, 0, c.st>>>(S.V, b, c.scal + 1, N);
  c.launches += 4;
  const double beta0 = read_scalar(c, c.scal);
  *iters = 0;
  if (!isfinite(beta0)) return MPM_ERR_NONFINITE;
  if (!(beta0 > 0.0)) return MPM_OK;
  const double target = rtol * beta0;
  int total = 0;
  bool converged = false;
  while (true) {
    int jc = 0;
    for (int j = 0; j < m; ++j) {
      T *Vj = S.V + (int64_t)j * N, *Zj = S.Z + (int64_t)j * N, *Vn = S.V + (int64_t)(j + 1) * N;
      precond<NB, T>(c, S, Vj, Zj);
      spmv<NB, T>(c, S, Zj, w);
      prof_begin(c, MPM_PROF_ORTH);
      {  // classical Gram-Schmidt, twice; the j + 1 products of a pass run side by side
        // slices per vector: enough blocks to stream the vectors at HBM speed
        // on large systems (about 8 elements per thread, up to NPART slices),
        // at least NPART / cnt on small ones; the update uses 1024-thread
        // blocks on large systems for the same reason (measured: slope
        // Gram-Schmidt 70 -> 46 ms per step; on the 62k-unknown footing the
        // larger blocks cost more than they gave, 1.4 -> 1.7 ms)
        const int cnt = j + 1;
        const int64_t by_size = N >= ORTH_BIG ? N / (TPB * 8) : 0;
        const int nbx = (int)std::min<int64_t>(NPART, std::max<int64_t>(std::max(16, NPART / cnt), by_size));
        const T *V = S.V, *wc = w;
        const double *ph = c.part;
        const int otpb = N >= ORTH_BIG ? ORTH_TPB : TPB;
        // FP64: the second pass only where the first lost the new direction's
        // digits (REORTH_THETA); FP32 always takes both passes
        const bool sel = sizeof(T) == sizeof(double);
        const double *skip = sel ? (const double *)(c.scal + 6) : nullptr;
        const int c1 = sel ? cnt + 1 : cnt;  // FP64: |w|^2 beside the products
        launch_pdl(c, k_multidot2<T>, dim3(nbx, c1), TPB, 0, V, wc, N, cnt, c.part, (const double *)nullptr);
        launch_pdl(c, k_multidot_reduce, c1, TPB, 0, ph, nbx, c1, h1, (const double *)nullptr);
        launch_pdl(c, k_orth_sub<T>, NPART, otpb, 0, w, V, (const double *)h1, cnt, N, c.part, sel ? 1 : 0,
                   (const double *)nullptr);
        if (sel)
          launch_pdl(c, k_reorth_test, 1, TPB, 0, ph, (int)NPART, (const double *)h1, cnt, REORTH_THETA,
                     c.scal + 6);
        launch_pdl(c, k_multidot2<T>, dim3(nbx, cnt), TPB, 0, V, wc, N, cnt, c.part, skip);
        launch_pdl(c, k_multidot_reduce, cnt, TPB, 0, ph, nbx, cnt, h2, skip);
        launch_pdl(c, k_orth_sub<T>, NPART, otpb, 0, w, V, (const double *)h2, cnt, N, c.part, 1, skip);
      }
      prof_end(c, MPM_PROF_ORTH);
      launch_pdl(c, k_arnoldi_finish, 1, TPB, 0, (const double *)c.part, (int)NPART, j, m, (const double *)h1,
                 (const double *)h2, c.H, c.gvec, c.cs, c.sn, c.scal);
      launch_pdl(c, k_scale_copy<T>, gN, TPB, 0, Vn, (const T *)w, (const double *)(c.scal + 1), N);
      ++total;
      jc = j + 1;
      const double res = read_scalar(c, c.scal);
      if (!isfinite(res)) return MPM_ERR_NONFINITE;
      if (res <= target) {
        converged = true;
        break;
      }
      if (total >= maxit) break;
    }
    k_backsolve<<<1, 32, 0, c.st>>>(c.H, c.gvec, jc, m, c.yv);
    k_update_x<T><<<gN, TPB, 0, c.st>>>(x, S.Z, c.yv, jc, N);
    c.launches += 2;
    if (converged || total >= maxit) break;
    // restart from the true residual r = b - A x (right preconditioning: x is
    // already in the unpreconditioned space)
    spmv<NB, T>(c, S, x, w);
    k_residual_vec<T><<<gN, TPB, 0, c.st>>>(w, b, N);
    k_dot_partial<T><<<NPART, TPB, 0, c.st>>>(w, w, N, c.part);
    k_reduce<<<1, TPB, 0, c.st>>>(c.part, NPART, c.scal + 2);
    k_gmres_init<<<1, 32, 0, c.st>>>(c.gvec, m, c.scal + 2, c.scal);
    k_scale_copy<T><<<gN, TPB, 0, c.st>>>(S.V, w, c.scal + 1, N);
    c.launches += 5;
    const double br = read_scalar(c, c.scal);
    if (!isfinite(br)) return MPM_ERR_NONFINITE;
    if (br <= target) {
      converged = true;
      break;
    }
  }
  *iters = total;
  if (check_cuda(c, cudaGetLastError(), "fgmres")) return MPM_ERR_CUDA;
  return converged ? MPM_OK : MPM_ERR_KRYLOV_STAGNATED;
}

template <typename T>
int dmalloc(T **p, int64_t n) {
  return cudaMalloc((void **)p, sizeof(T) * (size_t)(n > 0 ? n : 1)) == cudaSuccess ? MPM_OK
                                                                                     : MPM_ERR_NO_MEMORY;
}

}  // namespace

// ============================================================== launchers
int64_t scan_exclusive(Ctx &c, const int32_t *in, int32_t *out, int64_t n) {
  const int nb = (int)((n + SCAN_CHUNK - 1) / SCAN_CHUNK);
  if (nb > SCAN_CHUNK || nb > c.scan_cap) {
    c.last_error = "scan too long";
    return -1;
  }
  k_scan_blocks<<<nb, SCAN_T, 0, c.st>>>(in, out, n, c.scan_tmp);
  k_scan_top<<<1, SCAN_T, 0, c.st>>>(c.scan_tmp, nb);
  slot_reset(c, SLOT_SCAN);
  k_scan_add<<<nb, SCAN_T, 0, c.st>>>(out, n, c.scan_tmp, in, c.d_slot + SLOT_SCAN);
  c.launches += 3;
  double total;
  if (slot_wait(c, SLOT_SCAN, &total)) return -1;
  return (int64_t)llround(total);
}

int run_norm(Ctx &c, const double *x, double *norm) {
  slot_reset(c, SLOT_NORM);
  slot_reset(c, SLOT_ERR);
  k_dot_partial<double><<<NPART, TPB, 0, c.st>>>(x, x, c.N(), c.part);
  k_reduce_post<<<1, TPB, 0, c.st>>>(c.part, NPART, c.err, c.d_slot + SLOT_NORM, c.d_slot + SLOT_ERR);
  c.launches += 2;
  double n2, err;
  int rc = slot_wait(c, SLOT_NORM, &n2);
  if (!rc) rc = slot_wait(c, SLOT_ERR, &err);
  if (!rc) rc = dev_err_code(c, (int)err);
  *norm = sqrt(n2);
  return rc;
}

int read_dev_err(Ctx &c) {
  slot_reset(c, SLOT_WORD);
  k_post_err<<<1, 1, 0, c.st>>>(c.err, c.d_slot + SLOT_WORD);
  UPMPM_LAUNCH(c);
  double err;
  const int rc = slot_wait(c, SLOT_WORD, &err);
  return rc ? rc : dev_err_code(c, (int)err);
}

int batch_slices(Ctx &c, const std::vector<int32_t> &node_inst) {
  const int ni = c.ninst;
  std::vector<std::vector<int32_t>> of(ni + 1);  // nodes by instance; those between instances last
  for (size_t a = 0; a < node_inst.size(); ++a) of[node_inst[a] < 0 ? ni : node_inst[a]].push_back((int32_t)a);
  std::vector<int32_t> nodes, s0;
  std::vector<int4> sl;
  for (int i = 0; i <= ni; ++i) {
    s0.push_back((int32_t)sl.size());
    if (i == ni) c.bn_live = (int)sl.size();
    const int len = (int)of[i].size();
    for (int b = 0; b < len; b += BG_NODES)
      sl.push_back(make_int4(i < ni ? i : -1, (int)nodes.size() + b, std::min(BG_NODES, len - b), 0));
    nodes.insert(nodes.end(), of[i].begin(), of[i].end());
  }
  c.bn_all = (int)sl.size();
  if (dmalloc(&c.bn_nodes, nodes.size()) || dmalloc(&c.bn_s0, s0.size()) || dmalloc(&c.bn_slices, sl.size()) ||
      dmalloc(&c.bn_part, (int64_t)c.bn_live * PSTR) || dmalloc(&c.bn_npart, c.bn_live))
    return MPM_ERR_NO_MEMORY;
  cudaMemcpy(c.bn_nodes, nodes.data(), sizeof(int32_t) * nodes.size(), cudaMemcpyHostToDevice);
  cudaMemcpy(c.bn_s0, s0.data(), sizeof(int32_t) * s0.size(), cudaMemcpyHostToDevice);
  cudaMemcpy(c.bn_slices, sl.data(), sizeof(int4) * sl.size(), cudaMemcpyHostToDevice);
  return check_cuda(c, cudaGetLastError(), "node slices");
}

template <typename T>
int linsys_alloc(Ctx &c, LinSys<T> &S, bool krylov) {
  const int64_t nn = c.g.nnodes, N = c.N();
  const int nb = c.nb, m = c.m_restart;
  int rc = MPM_OK;
  auto A = [&](T **p, int64_t n) {
    if (!rc) rc = dmalloc(p, n);
  };
  A(&S.dscale, N);
  A(&S.dscinv, N);
  A(&S.dinv, nn * nb * nb);
  A(&S.rhs, N);
  A(&S.x, N);
  A(&S.w, N);
  if (krylov) {
    A(&S.V, (int64_t)(m + 1) * N);
    A(&S.Z, (int64_t)m * N);
  }
  if (!rc && c.opt.precond == MPM_PRECOND_SCHUR_MG) rc = schur_alloc<T>(c, S);
  return rc;
}

template <typename T>
void linsys_free(LinSys<T> &S) {
  schur_free<T>(S);
  T *ptrs[] = {S.val, S.dscale, S.dscinv, S.dinv, S.rhs, S.x, S.w, S.V, S.Z};
  for (T *p : ptrs)
    if (p) cudaFree(p);
  S.val = S.dscale = S.dscinv = S.dinv = S.rhs = S.x = S.w = S.V = S.Z = nullptr;
  S.cap = 0;
}

template <typename T>
int linsys_reserve(Ctx &c, LinSys<T> &S) {
  if (S.cap >= c.nnzb_cap && S.val) return MPM_OK;
  if (S.val) cudaFree(S.val);
  S.val = nullptr;
  S.cap = 0;
  if (step_malloc(c, (void **)&S.val, sizeof(T) * c.nnzb_cap * c.nb * c.nb)) {
    c.last_error = "device allocation of the block-CSR values failed";
    return MPM_ERR_NO_MEMORY;
  }
  S.cap = c.nnzb_cap;
  return MPM_OK;
}

template <typename T>
void run_scale_system(Ctx &c, LinSys<T> &S, const double *R) {
  const int64_t nn = c.g.nnodes;
  if (c.nb == 3)
    k_diag_scale<3, T><<<nblk(nn), TPB, 0, c.st>>>(nn, c.row_ptr, c.col, S.val, S.dscale, S.dscinv);
  else
    k_diag_scale<4, T><<<nblk(nn), TPB, 0, c.st>>>(nn, c.row_ptr, c.col, S.val, S.dscale, S.dscinv);
  k_scale_rhs<T><<<nblk(c.N()), TPB, 0, c.st>>>(c.N(), R, S.dscale, S.rhs);
  c.launches += 2;
}

template <typename T>
void run_add_solution(Ctx &c, const LinSys<T> &S, double *X) {
  k_add<T><<<nblk(c.N()), TPB, 0, c.st>>>(c.N(), X, S.x);
  UPMPM_LAUNCH(c);
}

template <typename T>
void run_to_scaled(Ctx &c, const LinSys<T> &S, T *z) {
  k_mul<T><<<nblk(c.N()), TPB, 0, c.st>>>(c.N(), z, S.dscinv);
  UPMPM_LAUNCH(c);
}

template <typename T>
void run_block_jacobi(Ctx &c, LinSys<T> &S) {
  const int64_t nn = c.g.nnodes;
  if (c.nb == 3)
    k_block_jacobi<3, T><<<nblk(nn), TPB, 0, c.st>>>(nn, c.row_ptr, c.col, S.val, S.dscale, S.dinv, c.err);
  else
    k_block_jacobi<4, T><<<nblk(nn), TPB, 0, c.st>>>(nn, c.row_ptr, c.col, S.val, S.dscale, S.dinv, c.err);
  UPMPM_LAUNCH(c);
}

template <typename T>
void run_precond(Ctx &c, LinSys<T> &S, const T *v, T *z) {
  if (c.nb == 3) precond<3, T>(c, S, v, z);
  else precond<4, T>(c, S, v, z);
}

template <typename T>
int run_fgmres(Ctx &c, LinSys<T> &S, double rtol, int maxit, int *iters) {
  if (c.nb == 3) return fgmres_impl<3, T>(c, S, rtol, maxit, iters);
  return fgmres_impl<4, T>(c, S, rtol, maxit, iters);
}

#define UPMPM_INST(T)                                                               \
  template int linsys_alloc<T>(Ctx &, LinSys<T> &, bool);                           \
  template void linsys_free<T>(LinSys<T> &);                                        \
  template int linsys_reserve<T>(Ctx &, LinSys<T> &);                               \
  template void run_scale_system<T>(Ctx &, LinSys<T> &, const double *);            \
  template void run_add_solution<T>(Ctx &, const LinSys<T> &, double *);            \
  template void run_to_scaled<T>(Ctx &, const LinSys<T> &, T *);                    \
  template void run_block_jacobi<T>(Ctx &, LinSys<T> &);                            \
  template void run_precond<T>(Ctx &, LinSys<T> &, const T *, T *);                 \
  template int run_fgmres<T>(Ctx &, LinSys<T> &, double, int, int *);
UPMPM_INST(double)
UPMPM_INST(float)
#undef UPMPM_INST

}  // namespace upmpm
