// mpm_mg_impl.cuh -- precision-generic body of mpm_mg.cu (included twice, with
// MG_REAL = double / float and MG_NS naming the namespace of that precision).

namespace MG_NS {
using real = MG_REAL;


constexpr int TPB = 256;
inline int nblk(int64_t n, int tpb = TPB) { return (int)((n + tpb - 1) / tpb); }

// Block size for a launch of `threads` threads: the largest of 256, 128, 64, 32
// that still gives two blocks per SM, so that small multigrid levels spread
// over the whole GPU (one SM's FP64 pipe is narrow; a level's rows packed into
// a few 256-thread blocks would run on a few SMs).
struct Geom {
  int blocks, tpb;
};
inline Geom geom(const Ctx &c, int64_t threads) {
  int t = 256;
  while (t > 32 && threads < (int64_t)t * 2 * c.nsm) t >>= 1;
  return {nblk(threads > 0 ? threads : 1, t), t};
}

// Thread maps of the set-up products: a tile of AP_ROWS rows takes all its slots
// before the next tile, a warp's lanes one slot in AP_ROWS consecutive rows.
constexpr int AP_ROWS = 32;
inline int64_t ap_threads(int64_t rows, int ns) { return (rows + AP_ROWS - 1) / AP_ROWS * AP_ROWS * ns; }

template <int D>
struct NS_ {
  static constexpr int v = D == 2 ? 25 : 125;
};

// Small dense inverse with partial pivoting (B <= 4); identity on failure.
template <int B>
__device__ inline bool invert_small(real A[B][B], real Inv[B][B]) {
  for (int i = 0; i < B; ++i)
    for (int j = 0; j < B; ++j) Inv[i][j] = i == j ? 1.0 : 0.0;
  for (int k = 0; k < B; ++k) {
    int piv = k;
    real best = fabs(A[k][k]);
    for (int i = k + 1; i < B; ++i)
      if (fabs(A[i][k]) > best) { best = fabs(A[i][k]); piv = i; }
    if (!(best > 1e-300)) {
      for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j) Inv[i][j] = i == j ? 1.0 : 0.0;
      return false;
    }
    if (piv != k)
      for (int j = 0; j < B; ++j) {
        real t = A[k][j]; A[k][j] = A[piv][j]; A[piv][j] = t;
        t = Inv[k][j]; Inv[k][j] = Inv[piv][j]; Inv[piv][j] = t;
      }
    const real inv = 1.0 / A[k][k];
    for (int j = 0; j < B; ++j) { A[k][j] *= inv; Inv[k][j] *= inv; }
    for (int i = 0; i < B; ++i) {
      if (i == k) continue;
      const real f = A[i][k];
      if (f == 0.0) continue;
      for (int j = 0; j < B; ++j) { A[i][j] -= f * A[k][j]; Inv[i][j] -= f * Inv[k][j]; }
    }
  }
  return true;
}

__device__ inline int find_col(const int32_t *__restrict__ col, int lo, int hi, int key) {
  hi -= 1;
  while (lo <= hi) {
    const int mid = (lo + hi) >> 1;
    const int c = col[mid];
    if (c == key) return mid;
    if (c < key) lo = mid + 1; else hi = mid - 1;
  }
  return -1;
}

// ------------------------------------------------------------ block split
// The blocks of the unscaled Jacobian in one pass: A (D x D), the compact B1
// (column D of the u rows) and B2 (row D of the u columns) where asked for, and
// in the fixed-stress approximation S = C plus the lumped term on the diagonal of
// free pressure rows (fsd; null otherwise).
template <int D>
__global__ void k_split_blocks(int64_t nnzb, const real *__restrict__ J, const int32_t *__restrict__ row_of,
                               const int32_t *__restrict__ col, const double *__restrict__ fsd,
                               const uint8_t *__restrict__ fixed, real *__restrict__ A, real *__restrict__ B1,
                               real *__restrict__ B2, real *__restrict__ S) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= nnzb) return;
  constexpr int NB = D + 1;
  alignas(16) real x[NB * NB];
  if constexpr (NB == 4) {  // a block is 64 or 128 bytes
    constexpr int W = 16 / (int)sizeof(real);
#pragma unroll
    for (int i = 0; i < 16 / W; ++i)
      reinterpret_cast<int4 *>(x)[i] = reinterpret_cast<const int4 *>(J + e * 16)[i];
  } else {
#pragma unroll
    for (int i = 0; i < NB * NB; ++i) x[i] = J[e * NB * NB + i];
  }
#pragma unroll
  for (int i = 0; i < D; ++i)
#pragma unroll
    for (int k = 0; k < D; ++k) A[e * D * D + i * D + k] = x[i * NB + k];
  if (B1)
#pragma unroll
    for (int k = 0; k < D; ++k) B1[e * D + k] = x[k * NB + D];
  if (B2)
#pragma unroll
    for (int k = 0; k < D; ++k) B2[e * D + k] = x[D * NB + k];
  if (fsd) {
    real s = x[D * NB + D];
    const int32_t a = row_of[e];
    if (col[e] == a && !fixed[(int64_t)a * NB + D]) s += (real)fsd[a];
    S[e] = s;
  }
}

// Block of row a coupling with node a + o, from the per-node coupling mask of
// the block sparsity (columns of a row are in mask-bit order); -1 if absent.
template <int D>
__device__ inline int mask_block(const uint64_t *__restrict__ mask, const int32_t *__restrict__ row_ptr,
                                 int a, int o0, int o1, int o2) {
  if (o0 < -3 || o0 > 3 || o1 < -3 || o1 > 3 || (D == 3 && (o2 < -3 || o2 > 3))) return -1;
  const int sl = (o0 + 3) + 7 * (o1 + 3) + (D == 3 ? 49 * (o2 + 3) : 0);
  const uint64_t *mk = mask + (int64_t)a * PATTERN_MASK_WORDS;
  const int w = sl >> 6;
  const uint64_t word = mk[w];
  if (!((word >> (sl & 63)) & 1ull)) return -1;
  int before = __popcll(word & ((1ull << (sl & 63)) - 1ull));
  for (int i = 0; i < w; ++i) before += __popcll(mk[i]);
  return row_ptr[a] + before;
}

__device__ inline void grid_xyz(const int nn0, const int nn1, int a, int c[3]) {
  const int r = a / nn0;
  c[0] = a - r * nn0;
  c[1] = r % nn1;
  c[2] = r / nn1;
}

// diag(A)_a^{-1} and the row sum of the B1 blocks of row a
template <int D>
__global__ void k_diag_inv_A(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, const real *__restrict__ A,
                             const real *__restrict__ B1, real *__restrict__ DAinv,
                             real *__restrict__ B1rs) {
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  const int e = find_col(col, row_ptr[a], row_ptr[a + 1], (int)a);
  real M[D][D], Inv[D][D];
  for (int i = 0; i < D; ++i)
    for (int k = 0; k < D; ++k) M[i][k] = e >= 0 ? A[(int64_t)e * D * D + i * D + k] : (i == k);
  invert_small<D>(M, Inv);
  for (int i = 0; i < D; ++i)
    for (int k = 0; k < D; ++k) DAinv[a * D * D + i * D + k] = Inv[i][k];
  real rs[D];
  for (int k = 0; k < D; ++k) rs[k] = 0.0;
  for (int eb = row_ptr[a]; eb < row_ptr[a + 1]; ++eb)
    for (int k = 0; k < D; ++k) rs[k] += B1[(int64_t)eb * D + k];
  for (int k = 0; k < D; ++k) B1rs[a * D + k] = rs[k];
}

// W_ac = B2_ac diag(A)_c^{-1} (a 1 x D row per block)
template <int D>
__global__ void k_schur_w(int64_t nnzb, const int32_t *__restrict__ col, const real *__restrict__ J,
                          const real *__restrict__ DAinv, real *__restrict__ W) {
  const int64_t ec = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (ec >= nnzb) return;
  constexpr int NB = D + 1;
  const int64_t c = col[ec];
  for (int k = 0; k < D; ++k) {
    real w = 0.0;
    for (int i = 0; i < D; ++i) w += J[ec * NB * NB + D * NB + i] * DAinv[c * D * D + i * D + k];
    W[ec * D + k] = w;
  }
}

// S_ab = C_ab - sum_c W_ac B1_cb on J's sparsity, one thread per block (a, b),
// mapped as k_mg_ap (a tile of rows takes all offsets, a warp's lanes share one).
// Row a's blocks are walked by the bits of its coupling mask (ascending, like
// its columns), so that c and its offset to b come from the bit alone; (c, b) is
// found from c's mask.  (Reading col[ec] and dividing for c's coordinates, the
// set-up of 64 batched footings took 5.2 ms against 2.7.)
template <int D>
__global__ void k_schur_rows(int nn0, int nn1, int64_t nnodes, const uint64_t *__restrict__ mask,
                             const int32_t *__restrict__ row_ptr, const real *__restrict__ J,
                             const real *__restrict__ B1, const real *__restrict__ W, real *__restrict__ S) {
  constexpr int NB = D + 1, NSL = D == 2 ? 49 : 343;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t tile = t / (AP_ROWS * NSL);
  const int rem = (int)(t - tile * (AP_ROWS * NSL));
  const int64_t ar = tile * AP_ROWS + rem % AP_ROWS;
  if (ar >= nnodes) return;
  const int a = (int)ar, sl = rem / AP_ROWS;
  const int o0 = sl % 7 - 3, o1 = (sl / 7) % 7 - 3, o2 = D == 3 ? sl / 49 - 3 : 0;
  const int eb = mask_block<D>(mask, row_ptr, a, o0, o1, o2);
  if (eb < 0) return;
  real prod = 0.0;
  int ec = row_ptr[a];
  for (int w = 0; w < (D == 2 ? 1 : PATTERN_MASK_WORDS); ++w)
    for (uint64_t bits = mask[(int64_t)a * PATTERN_MASK_WORDS + w]; bits; bits &= bits - 1, ++ec) {
      const int sc = 64 * w + __ffsll((long long)bits) - 1;
      const int c0 = sc % 7 - 3, c1 = (sc / 7) % 7 - 3, c2 = D == 3 ? sc / 49 - 3 : 0;
      const int cn = a + c0 + nn0 * (c1 + nn1 * c2);
      const int e_cb = mask_block<D>(mask, row_ptr, cn, o0 - c0, o1 - c1, o2 - c2);
      if (e_cb < 0) continue;
      for (int k = 0; k < D; ++k) prod += W[(int64_t)ec * D + k] * B1[(int64_t)e_cb * D + k];
    }
  S[eb] = J[(int64_t)eb * NB * NB + D * NB + D] - prod;
}

// The part of row a's full product sum_c W_ac (sum_b B1_cb) that fell outside
// the sparsity is added to S_aa.
template <int D>
__global__ void k_schur_lump(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, const real *__restrict__ J,
                             const real *__restrict__ W, const real *__restrict__ B1rs,
                             real *__restrict__ S) {
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  constexpr int NB = D + 1;
  real total = 0.0, kept = 0.0;
  int diag = -1;
  for (int e = row_ptr[a]; e < row_ptr[a + 1]; ++e) {
    const int cn = col[e];
    if (cn == a) diag = e;
    for (int k = 0; k < D; ++k) total += W[(int64_t)e * D + k] * B1rs[(int64_t)cn * D + k];
    kept += J[(int64_t)e * NB * NB + D * NB + D] - S[e];
  }
  if (diag >= 0) S[diag] -= (total - kept);
}

// ------------------------------------------------------------ Schur apply
// The Krylov solver works on D J D (D = dsc); the blocks below are the
// unscaled physical ones, so the preconditioner of D J D is D^-1 M^-1 D^-1.  The
// split applies the right D^-1 (dsi = |diag J|^{1/2}, stored: products instead of
// FP64 divisions, which run long on the narrow FP64 pipe); the left one is left
// out: z = M^-1 D^-1 v, the vector in the unscaled unknowns that the product
// y = D J z and the solution take.
// v_u, v_p of the unscaled system; v_p is the S-cycle's level-0 rhs, whose
// first smoothing sweep from zero (x = omega Dinv b, pointwise) is done here.
template <int D>
__global__ void k_split(int64_t nnodes, const real *__restrict__ v, const real *__restrict__ dsi,
                        real *__restrict__ vu, real *__restrict__ bs0, real *__restrict__ xs0,
                        const real *__restrict__ dinvs0, real omega) {
  pdl_enter();
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  for (int k = 0; k < D; ++k) vu[a * D + k] = v[a * (D + 1) + k] * dsi[a * (D + 1) + k];
  const real vp = v[a * (D + 1) + D] * dsi[a * (D + 1) + D];
  bs0[a] = vp;
  xs0[a] = omega * (dinvs0[a] * vp);
}

// Lower-triangular order: v_u is the A-cycle's level-0 rhs, with its first
// smoothing sweep from zero (x = omega Dinv_A v_u, a D x D block per node);
// v_p is kept for the S-cycle's rhs v_p - B2 z_u.
template <int D>
__global__ void k_split_lower(int64_t nnodes, const real *__restrict__ v, const real *__restrict__ dsi,
                              real *__restrict__ ba0, real *__restrict__ xa0, const real *__restrict__ dinva0,
                              real *__restrict__ vp, real omega) {
  pdl_enter();
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  real vu[D];
  for (int k = 0; k < D; ++k) {
    vu[k] = v[a * (D + 1) + k] * dsi[a * (D + 1) + k];
    ba0[a * D + k] = vu[k];
  }
  for (int i = 0; i < D; ++i) {
    real sv = 0.0;
    for (int j = 0; j < D; ++j) sv = fma(dinva0[a * D * D + i * D + j], vu[j], sv);
    xa0[a * D + i] = omega * sv;
  }
  vp[a] = v[a * (D + 1) + D] * dsi[a * (D + 1) + D];
}

// w_u = v_u - B1 z_p with the compact unscaled B1: the A-cycle's level-0 rhs,
// with its first smoothing sweep from zero (x = omega Dinv w_u).  LN lanes per
// row (LN_ below).
template <int D, int LN>
__global__ void k_b1c_update(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, const real *__restrict__ B1,
                             const real *__restrict__ zp, const real *__restrict__ vu,
                             real *__restrict__ ba0, real *__restrict__ xa0,
                             const real *__restrict__ dinva0, real omega) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t a = t / LN;
  const int lane = (int)(t % LN);
  const bool valid = a < nnodes;
  real acc[D];
  for (int k = 0; k < D; ++k) acc[k] = 0;
  if (valid) {
    const int e1 = row_ptr[a + 1];
    for (int e = row_ptr[a] + lane; e < e1; e += LN) {
      const real z = zp[col[e]];
      for (int k = 0; k < D; ++k) acc[k] = fma(B1[(int64_t)e * D + k], z, acc[k]);
    }
  }
  for (int o = LN / 2; o > 0; o >>= 1)
    for (int k = 0; k < D; ++k) acc[k] += __shfl_xor_sync(0xffffffffu, acc[k], o);
  if (!valid || lane >= D) return;
  // lane i < D finishes component i
  real s = 0.0, wi = 0.0;
  for (int j = 0; j < D; ++j) {
    const real wj = vu[a * D + j] - acc[j];
    wi = lane == j ? wj : wi;
    s = fma(dinva0[a * D * D + lane * D + j], wj, s);
  }
  ba0[a * D + lane] = wi;
  xa0[a * D + lane] = omega * s;
}

template <int D, int LN>
__global__ void k_b2c_update(int64_t nnodes, const int32_t *__restrict__ row_ptr,
                             const int32_t *__restrict__ col, const real *__restrict__ B2,
                             const real *__restrict__ zu, const real *__restrict__ vp,
                             real *__restrict__ bs0, real *__restrict__ xs0,
                             const real *__restrict__ dinvs0, real omega) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t a = t / LN;
  const int lane = (int)(t % LN);
  const bool valid = a < nnodes;
  real acc = 0;
  if (valid) {
    const int e1 = row_ptr[a + 1];
    for (int e = row_ptr[a] + lane; e < e1; e += LN) {
      const int64_t b = col[e];
      for (int k = 0; k < D; ++k) acc = fma(B2[(int64_t)e * D + k], zu[b * D + k], acc);
    }
  }
  for (int o = LN / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (!valid || lane != 0) return;
  const real w = vp[a] - acc;
  bs0[a] = w;
  xs0[a] = omega * (dinvs0[a] * w);
}

template <int D>
__global__ void k_merge(int64_t nnodes, const real *__restrict__ zu, const real *__restrict__ zp,
                        real *__restrict__ z) {
  pdl_enter();
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= nnodes) return;
  for (int k = 0; k < D; ++k) z[a * (D + 1) + k] = zu[a * D + k];
  z[a * (D + 1) + D] = zp[a];
}

// ------------------------------------------------------------ multigrid
struct LevelDev {
  int nn[3];
  int64_t nnodes;
  const int32_t *row_ptr, *col;  // level 0 only
  const real *val;              // level 0: block-CSR values
  real *sval;                   // coarse levels: dense 5^d stencil values
  uint8_t *nslot;               // coarse levels: nonzero blocks of each row (0: a node without coupling)
  real *dinv;
  // level 0 only: Dirichlet / inactive DOFs are left out of the transfers
  const uint8_t *fixed;           // fixed[a * mstride + moff + i] != 0: DOF fixed
  int mstride, moff;
  const uint64_t *mask;           // level 0 only: coupling mask of the block sparsity
  // instance of every node (-1 between instances): the transfers connect a
  // fine and a coarse node only within one instance, so the hierarchy of a
  // batched context never mixes instances (null for a single instance)
  const int32_t *inst;
};

__device__ inline real free_w(const LevelDev &L, int64_t a, int i) {
  return (L.fixed && L.fixed[a * L.mstride + L.moff + i]) ? 0.0 : 1.0;
}

// Lanes per row of the row kernels (a row is one node: up to 49 blocks of the
// fine block-CSR in 2D, 125 in 3D, 5^d slots of a coarse stencil).  Eight
// lanes keep the shuffle reduction (log2 LN steps per block row) small next to
// the row's FMAs on GB300's narrow FP64 pipe; FP32 3D rows take 16 (latency).
// Large FP64 levels take 4 lanes: on the FP64 pipe a warp instruction costs the
// same with any number of lanes, and 4 lanes spend fewer of them on a row's
// reduction, epilogue and last partial round: one application on the 4.2M-point
// slope 4.9 -> 4.4 ms, on 64 batched columns 389 -> 333 us (both with the branch-free
// restriction below).
template <int D>
struct LN_ {
  static constexpr int v = (sizeof(real) == sizeof(double) || D == 2) ? 8 : 16;
  static constexpr int large = sizeof(real) == sizeof(double) ? 4 : v;
  // small 3D levels: a row of up to 125 blocks on one warp, since what bounds
  // them is the chain of a lane's blocks (480 nodes: 22-28 -> 11 us a pass; 3,135:
  // 22-28 -> 15)
  static constexpr int small = D == 3 ? 32 : v;
  // 3D levels between: their rows (100 blocks) are bound by FP64 issue too (24k nodes:
  // 16 lanes 75-79 us a pass, 8 lanes 62-66, 4 lanes 63)
  static constexpr int mid = D == 3 && sizeof(real) == sizeof(double) ? 4 : v;
};
constexpr int64_t LN_LARGE_ROWS = 1 << 16, LN_SMALL_ROWS = 1 << 13;
// f(lanes) with the compile-time lane count for a level of so many rows
template <int D, typename F>
inline void with_lanes(int64_t rows, F &&f) {
  if (rows >= LN_LARGE_ROWS) f(std::integral_constant<int, LN_<D>::large>{});
  else if (rows < LN_SMALL_ROWS) f(std::integral_constant<int, LN_<D>::small>{});
  else f(std::integral_constant<int, LN_<D>::mid>{});
}

// Component `lane` (< B) of a B-vector held in registers, without indexing
// the register array by a run-time value.
template <int B>
__device__ inline real pick(const real v[B], int lane) {
  real o = v[0];
#pragma unroll
  for (int i = 1; i < B; ++i) o = lane == i ? v[i] : o;
  return o;
}

// Partial sum over the blocks of row a handled by `lane` (of LN lanes):
// acc += A_ab x_b, one FMA per matrix value.
template <int B, int D, bool ST, int LN>
__device__ inline void row_partial(const LevelDev &L, int64_t a, int lane, const real *__restrict__ x,
                                   real acc[B]) {
  if (!ST) {
    const int e1 = L.row_ptr[a + 1];
    for (int e = L.row_ptr[a] + lane; e < e1; e += LN) {
      const int64_t b = L.col[e];
      const real *blk = L.val + (int64_t)e * B * B;
      real xb[B];
      for (int j = 0; j < B; ++j) xb[j] = x[b * B + j];
      for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j) acc[i] = fma(blk[i * B + j], xb[j], acc[i]);
    }
  } else {
    int ac[3];
    grid_xyz(L.nn[0], L.nn[1], (int)a, ac);
    constexpr int NS = NS_<D>::v;
    const real *base = L.sval + a * NS * B * B;
    // rows without coupling (grid nodes outside the material: half of the
    // slope's coarse grids) are skipped whole
    if (L.nslot[a] == 0) return;
#pragma unroll 16
    for (int k = 0; k < (NS + LN - 1) / LN; ++k) {
      const int s = lane + k * LN;
      const int o0 = s % 5 - 2, o1 = (s / 5) % 5 - 2, o2 = D == 3 ? s / 25 - 2 : 0;
      const int b0 = ac[0] + o0, b1 = ac[1] + o1, b2 = ac[2] + o2;
      if (s >= NS || b0 < 0 || b0 >= L.nn[0] || b1 < 0 || b1 >= L.nn[1] || b2 < 0 || b2 >= L.nn[2]) continue;
      const int64_t b = b0 + L.nn[0] * (b1 + L.nn[1] * b2);
      const real *blk = base + s * B * B;
      real xb[B];
      for (int j = 0; j < B; ++j) xb[j] = x[b * B + j];
      for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j) acc[i] = fma(blk[i * B + j], xb[j], acc[i]);
    }
  }
}

template <int B, int LN>
__device__ inline void lane_reduce(real acc[B]) {
  for (int o = LN / 2; o > 0; o >>= 1)
    for (int i = 0; i < B; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
}

template <int B, int D, bool ST>
__global__ void k_mg_dinv(LevelDev L, int *err) {
  const int64_t a = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (a >= L.nnodes) return;
  real M[B][B], Inv[B][B];
  for (int i = 0; i < B; ++i)
    for (int j = 0; j < B; ++j) M[i][j] = (i == j) ? 1.0 : 0.0;
  if (!ST) {
    const int e = find_col(L.col, L.row_ptr[a], L.row_ptr[a + 1], (int)a);
    if (e >= 0)
      for (int i = 0; i < B; ++i)
        for (int j = 0; j < B; ++j) M[i][j] = L.val[(int64_t)e * B * B + i * B + j];
  } else {
    constexpr int NS = NS_<D>::v;
    const int s = D == 2 ? 12 : 62;  // centre slot of the 5^d stencil
    for (int i = 0; i < B; ++i)
      for (int j = 0; j < B; ++j) M[i][j] = L.sval[(a * NS + s) * B * B + i * B + j];
  }
  if (!invert_small<B>(M, Inv)) {
    // an all-zero diagonal block (e.g. a node without coupling) acts as identity
    for (int i = 0; i < B; ++i)
      for (int j = 0; j < B; ++j) Inv[i][j] = i == j ? 1.0 : 0.0;
  }
  for (int i = 0; i < B; ++i)
    for (int j = 0; j < B; ++j) L.dinv[a * B * B + i * B + j] = Inv[i][j];
}

// One damped block-Jacobi sweep: xo = xi + w Dinv (b - A xi); zero_init: xi = 0.
// LN lanes per row.
template <int B, int D, bool ST, int LN>
__global__ void k_mg_smooth(LevelDev L, const real *__restrict__ xi, real *__restrict__ xo,
                            const real *__restrict__ b, real omega, int zero_init) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t a = t / LN;
  const int lane = (int)(t % LN);
  const bool valid = a < L.nnodes;
  real ax[B];
  for (int i = 0; i < B; ++i) ax[i] = 0.0;
  if (valid && !zero_init) row_partial<B, D, ST, LN>(L, a, lane, xi, ax);
  lane_reduce<B, LN>(ax);  // every lane of the row now holds (A xi)_a
  if (!valid || lane >= B) return;
  // lane i < B finishes component i: B FMAs of row i of Dinv
  real s = 0.0;
  for (int j = 0; j < B; ++j) s = fma(L.dinv[a * B * B + lane * B + j], b[a * B + j] - ax[j], s);
  xo[a * B + lane] = (zero_init ? 0.0 : xi[a * B + lane]) + omega * s;
}

// Fine (block-CSR) level with B <= 2, a group of GS = B * SPL lanes per row:
// lane (r, part) sums block row r over the row's blocks part, part + SPL, ...
// (one FMA per stored value, all lanes busy), one shuffle sum over the SPL
// parts gives (A x)_r, and for a sweep the row's B residuals are exchanged
// inside the group: out = b - A x (residual) or x + omega Dinv (b - A x).
template <int B, int SPL, bool SMOOTH>
__global__ void k_mg_csr_row(LevelDev L, const real *__restrict__ x, real *__restrict__ out,
                             const real *__restrict__ b, real omega) {
  pdl_enter();
  constexpr int GS = B * SPL;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t a = t / GS;
  const int lg = (int)(t - a * GS);
  const int r = lg / SPL, part = lg - r * SPL;
  const bool valid = a < L.nnodes;
  real acc = 0;
  if (valid) {
    const int e1 = L.row_ptr[a + 1];
#pragma unroll 4
    for (int e = L.row_ptr[a] + part; e < e1; e += SPL) {
      const real *blk = L.val + (int64_t)e * B * B + r * B;
      const real *xb = x + (int64_t)L.col[e] * B;
#pragma unroll
      for (int c = 0; c < B; ++c) acc = fma(blk[c], xb[c], acc);
    }
  }
#pragma unroll
  for (int o = SPL / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  const real res = valid ? b[a * B + r] - acc : real(0);
  if (!SMOOTH) {
    if (valid && part == 0) out[a * B + r] = res;
    return;
  }
  const int base = (int)(threadIdx.x & 31) - lg;
  real rv[B];
#pragma unroll
  for (int c = 0; c < B; ++c) rv[c] = __shfl_sync(0xffffffffu, res, base + c * SPL);
  if (!valid || part != 0) return;
  real sum = 0;
#pragma unroll
  for (int c = 0; c < B; ++c) sum = fma(L.dinv[a * B * B + r * B + c], rv[c], sum);
  out[a * B + r] = x[a * B + r] + omega * sum;
}

template <int B, int D, bool ST, int LN>
__global__ void k_mg_resid(LevelDev L, const real *__restrict__ x, const real *__restrict__ b,
                           real *__restrict__ r) {
  pdl_enter();
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t a = t / LN;
  const int lane = (int)(t % LN);
  const bool valid = a < L.nnodes;
  real ax[B];
  for (int i = 0; i < B; ++i) ax[i] = 0.0;
  if (valid) row_partial<B, D, ST, LN>(L, a, lane, x, ax);
  lane_reduce<B, LN>(ax);
  if (!valid || lane >= B) return;
  r[a * B + lane] = b[a * B + lane] - pick<B>(ax, lane);
}

// ---- coarsest level: exact solve with a dense inverse built at set-up
// Dense copy of the coarsest operator (n = nnodes * B unknowns).
template <int B, int D, bool ST>
__global__ void k_dense_fill(LevelDev L, real *__restrict__ Ad) {
  const int64_t n = L.nnodes * B;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int64_t ri = t / n, ci = t % n;
  const int64_t a = ri / B, b = ci / B;
  const int i = (int)(ri % B), j = (int)(ci % B);
  real v = 0.0;
  if (!ST) {
    const int e = find_col(L.col, L.row_ptr[a], L.row_ptr[a + 1], (int)b);
    if (e >= 0) v = L.val[(int64_t)e * B * B + i * B + j];
  } else {
    int ac[3], bc[3];
    ac[0] = (int)(a % L.nn[0]); ac[1] = (int)((a / L.nn[0]) % L.nn[1]); ac[2] = (int)(a / ((int64_t)L.nn[0] * L.nn[1]));
    bc[0] = (int)(b % L.nn[0]); bc[1] = (int)((b / L.nn[0]) % L.nn[1]); bc[2] = (int)(b / ((int64_t)L.nn[0] * L.nn[1]));
    const int o0 = bc[0] - ac[0], o1 = bc[1] - ac[1], o2 = bc[2] - ac[2];
    if (o0 >= -2 && o0 <= 2 && o1 >= -2 && o1 <= 2 && o2 >= -2 && o2 <= 2) {
      constexpr int NS = NS_<D>::v;
      const int sl = (o0 + 2) + 5 * (o1 + 2) + (D == 3 ? 25 * (o2 + 2) : 0);
      v = L.sval[(a * NS + sl) * B * B + i * B + j];
    }
  }
  Ad[t] = v;
}

// Inverse of the dense coarsest operator Ad (n x n, row-major) into Ai, for
// the two hierarchies side by side (job 0, job 1), in two kernels:
//   k_dense_lu: LU factorisation with partial pivoting, one block per job (in
//     dynamic shared memory when it fits), row interchanges in piv[k] (LAPACK
//     order), n^3 / 3 FMAs; the transpose of the factors, with the reciprocals of
//     the diagonal, into At;
//   k_dense_inv_cols: column c of the inverse from P A = L U (forward and back
//     substitution on e_c), a warp per column with the vector in registers, so
//     the n^3 FMAs of the inverse spread over many SMs.
// Both are chains of n steps, and what a step costs is its barriers and the FP64
// instructions on its path: the pivot is found by one warp comparing magnitudes
// as integers, the elimination takes a warp per row, and the substitutions need
// no barrier (n = 72 and 36: 306 + 64 -> 153 + 36 us; n = 180 and 60: 1,380 + 191 ->
// 1,175 + 153, half of it the FP64 work of one SM).
// Columns with no usable pivot (below 1e-14 of the largest entry: nodes
// without material on the coarsest grid) are singular directions: their
// unknowns get zero in every column of the inverse, so the coarse correction
// leaves them alone.
struct DenseJob {
  int n;
  real *Ad, *Ai, *At;
  int *piv;  // n: row interchanged with row k, -1 marks a singular column; n: P's column c has its 1 here
};

constexpr int DENSE_LU_THREADS = 512;
constexpr size_t DENSE_SMEM_MAX = 220 * 1024;

// bits of |v|, which order as the magnitudes do (NaN above all)
__device__ __forceinline__ unsigned long long mag_bits(double v) {
  return (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
}
__device__ __forceinline__ unsigned long long mag_bits(float v) {
  return (unsigned long long)(__float_as_uint(v) & 0x7fffffffu);
}

// ns: the trailing ns x ns part of a job is factorised in shared memory (all of
// it when n <= ns), the columns before it in place in Ad
__global__ void __launch_bounds__(DENSE_LU_THREADS) k_dense_lu(DenseJob j0, DenseJob j1, int ns) {
  const DenseJob job = blockIdx.x == 0 ? j0 : j1;
  const int n = job.n, base = n > ns ? n - ns : 0;
  __shared__ int piv;
  __shared__ real rpiv;
  __shared__ int spiv[1024];
  __shared__ unsigned long long red[DENSE_LU_THREADS / 32];
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  real *Ms = reinterpret_cast<real *>(dyn_smem);
  const int lds = (n - base) | 1;  // odd: a column's entries in different banks
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned long long top = 0;  // largest magnitude, for the singular-pivot threshold
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) top = max(top, mag_bits(job.Ad[t]));
  for (int o = 16; o > 0; o >>= 1) top = max(top, __shfl_xor_sync(0xffffffffu, top, o));
  if (lane == 0) red[wid] = top;
  __syncthreads();
  for (int i = 0; i < nw; ++i) top = max(top, red[i]);
  const real amax = sizeof(real) == 8 ? (real)__longlong_as_double((long long)top)
                                      : (real)__uint_as_float((unsigned)top);
  // columns k0 .. k1 - 1 of the matrix M (leading dimension ld, entry (o, o) first)
  auto columns = [&](real *M, int ld, int o, int k0, int k1) {
    for (int k = k0; k < k1; ++k) {
      if (wid == 0) {  // pivot: largest |M[i][k]|, i >= k, the first of equals
        unsigned long long best = 0;
        int bi = n;
        for (int i = k + lane; i < n; i += 32) {
          const unsigned long long v = mag_bits(M[(i - o) * ld + k - o]);
          if (v > best || bi == n) { best = v; bi = i; }
        }
        for (int q = 16; q > 0; q >>= 1) {
          const unsigned long long ov = __shfl_xor_sync(0xffffffffu, best, q);
          const int oi = __shfl_xor_sync(0xffffffffu, bi, q);
          if (oi < n && (bi == n || ov > best || (ov == best && oi < bi))) { best = ov; bi = oi; }
        }
        if (lane == 0) {
          const real v = M[(bi - o) * ld + k - o];
          const bool use = fabs(v) > real(1e-14) * amax;
          piv = spiv[k] = use ? bi : -1;
          rpiv = use ? real(1) / v : real(0);
          job.piv[k] = piv;
          job.At[(int64_t)k * n + k] = rpiv;
        }
      }
      __syncthreads();
      const int p = piv;
      const real inv = rpiv;
      if (p < 0) {  // singular column: no elimination, zero multipliers
        for (int i = k + 1 + threadIdx.x; i < n; i += blockDim.x) M[(i - o) * ld + k - o] = 0;
        __syncthreads();
        continue;
      }
      if (p != k) {  // (the multipliers of the columns before o are in Ad)
        for (int j = threadIdx.x; j < n; j += blockDim.x) {
          real *a = j < o ? job.Ad + (int64_t)k * n + j : M + (k - o) * ld + j - o;
          real *b = j < o ? job.Ad + (int64_t)p * n + j : M + (p - o) * ld + j - o;
          const real t1 = *a;
          *a = *b;
          *b = t1;
        }
        __syncthreads();
      }
      const real *row = M + (k - o) * ld - o;
      for (int i = k + 1 + wid; i < n; i += nw) {
        real *mi = M + (i - o) * ld - o;
        const real l = mi[k] * inv;
        for (int j = k + 1 + lane; j < n; j += 32) mi[j] = fma(-l, row[j], mi[j]);
        __syncwarp();
        if (lane == 0) mi[k] = l;
      }
      __syncthreads();
    }
  };
  columns(job.Ad, n, 0, 0, base);
  for (int t = threadIdx.x; t < (n - base) * (n - base); t += blockDim.x) {
    const int i = t / (n - base), j = t % (n - base);
    Ms[i * lds + j] = job.Ad[(int64_t)(i + base) * n + j + base];
  }
  __syncthreads();
  columns(Ms, lds, base, base, n);
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int i = t % n, k = t / n;  // At[k][i] = M[i][k] off the diagonal
    if (i != k) job.At[t] = i >= base && k >= base ? Ms[(i - base) * lds + k - base] : job.Ad[(int64_t)i * n + k];
  }
  for (int c = threadIdx.x; c < n; c += blockDim.x) {  // where the interchanges take entry c of e_c
    int pos = c;
    for (int k = 0; k < n; ++k) {
      const int p = spiv[k];
      if (p >= 0) pos = pos == k ? p : (pos == p ? k : pos);
    }
    job.piv[n + c] = pos;
  }
}

// warp (c, job): column c of the job's inverse, n <= 32 NR; the factors' columns
// are fetched PF steps ahead (they do not depend on the vector)
template <int NR, int PF>
__device__ void dense_inv_col(const DenseJob &job, int c, int lane) {
  const int n = job.n;
  const real *At = job.At;
  const int pos = job.piv[n + c];
  real y[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) y[r] = lane + 32 * r == pos ? real(1) : real(0);
  auto entry = [&](int i) {  // y_i
    real v = y[0];
#pragma unroll
    for (int r = 1; r < NR; ++r) v = (i >> 5) == r ? y[r] : v;
    return __shfl_sync(0xffffffffu, v, i & 31);
  };
  real cur[PF][NR], nxt[PF][NR], dc[PF], dn[PF];
  // L y = P e_c (unit lower triangle), by columns
  auto fetch_l = [&](int i0, real (&a)[PF][NR]) {
#pragma unroll
    for (int u = 0; u < PF; ++u)
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int i = i0 + u, k = lane + 32 * r;
        a[u][r] = i < n && k > i && k < n ? At[(int64_t)i * n + k] : real(0);
      }
  };
  fetch_l(0, cur);
  for (int i0 = 0; i0 < n; i0 += PF) {
    fetch_l(i0 + PF, nxt);
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      if (i0 + u >= n) break;
      const real yi = entry(i0 + u);
#pragma unroll
      for (int r = 0; r < NR; ++r) y[r] = fma(-cur[u][r], yi, y[r]);
    }
#pragma unroll
    for (int u = 0; u < PF; ++u)
#pragma unroll
      for (int r = 0; r < NR; ++r) cur[u][r] = nxt[u][r];
  }
  // U x = y, by columns from the last
  auto fetch_u = [&](int i0, real (&a)[PF][NR], real (&dg)[PF]) {
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      const int i = i0 - u;
      dg[u] = i >= 0 ? At[(int64_t)i * n + i] : real(0);
#pragma unroll
      for (int r = 0; r < NR; ++r) a[u][r] = i >= 0 && lane + 32 * r < i ? At[(int64_t)i * n + lane + 32 * r] : real(0);
    }
  };
  fetch_u(n - 1, cur, dc);
  for (int i0 = n - 1; i0 >= 0; i0 -= PF) {
    fetch_u(i0 - PF, nxt, dn);
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      const int i = i0 - u;
      if (i < 0) break;
      const real xi = entry(i) * dc[u];
#pragma unroll
      for (int r = 0; r < NR; ++r) y[r] = lane + 32 * r == i ? xi : fma(-cur[u][r], xi, y[r]);
    }
#pragma unroll
    for (int u = 0; u < PF; ++u) {
      dc[u] = dn[u];
#pragma unroll
      for (int r = 0; r < NR; ++r) cur[u][r] = nxt[u][r];
    }
  }
#pragma unroll
  for (int r = 0; r < NR; ++r)
    if (lane + 32 * r < n) job.Ai[(int64_t)(lane + 32 * r) * n + c] = y[r];
}

__global__ void __launch_bounds__(128) k_dense_inv_cols(DenseJob j0, DenseJob j1) {
  const DenseJob job = blockIdx.y == 0 ? j0 : j1;
  const int c = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= job.n) return;
  if (job.n <= 96) dense_inv_col<3, 8>(job, c, lane);
  else if (job.n <= 192) dense_inv_col<6, 4>(job, c, lane);
  else dense_inv_col<32, 1>(job, c, lane);
}

// x = Ai b
// one warp per row i; lanes split the row and reduce
__global__ void k_dense_apply(int n, const real *__restrict__ Ai, const real *__restrict__ b,
                              real *__restrict__ x) {
  pdl_enter();
  const int i = (int)((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  real s = 0.0;
  if (i < n) {
    const real *row = Ai + (int64_t)i * n;
#pragma unroll 8
    for (int j = lane; j < n; j += 32) s = fma(row[j], b[j], s);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (i < n && lane == 0) x[i] = s;
}

// weight of coarse node I for fine node a along one axis
__device__ inline real pw(int a, int I) {
  const int dlt = a - 2 * I;
  return dlt == 0 ? 1.0 : ((dlt == 1 || dlt == -1) ? 0.5 : 0.0);
}

// b_c(I) = sum_a P_aI r_a over the fine nodes within one fine cell of 2I; if
// xc is given, also the coarse level's first smoothing sweep from zero,
// x_c = omega Dinv_c b_c.  A lane per component (32 / B nodes a warp).  All
// children's loads without branches between them (a child outside the grid, of
// another instance or fixed contributes a selected zero), so that the loads of
// the 3^d children are in flight together: one application on the 80k-point
// footing 112 -> 104 us (a third of its kernels restrict); a lane per component
// instead of per node: 16 -> 10 and 12 -> 7 us a launch on 3D levels of 3,135 and 480
// nodes.
template <int B>
__host__ __device__ constexpr int restrict_nodes() { return 32 / B; }  // per warp
template <int B, int D>
__global__ void k_mg_restrict(LevelDev F, LevelDev Cl, const real *__restrict__ rf,
                              real *__restrict__ bc, real *__restrict__ xc, real omega) {
  pdl_enter();
  constexpr int NPW = restrict_nodes<B>();
  const int lane = threadIdx.x & 31;
  const int64_t I = ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5) * NPW + lane / B;
  const int i = lane % B;
  const bool live = lane < NPW * B && I < Cl.nnodes;
  real acc = 0;
  if (live) {
    int Ic[3];
    grid_xyz(Cl.nn[0], Cl.nn[1], (int)I, Ic);
    const int inst_c = Cl.inst ? Cl.inst[I] : 0;
#pragma unroll
    for (int ch = 0; ch < (D == 3 ? 27 : 9); ++ch) {
      const int d0 = ch % 3 - 1, d1 = ch / 3 % 3 - 1, d2 = D == 3 ? ch / 9 - 1 : 0;
      const int a0 = 2 * Ic[0] + d0, a1 = 2 * Ic[1] + d1, a2 = 2 * Ic[2] + d2;
      const bool in = a0 >= 0 && a0 < F.nn[0] && a1 >= 0 && a1 < F.nn[1] && (D == 2 || (a2 >= 0 && a2 < F.nn[2]));
      const int64_t a = in ? a0 + (int64_t)F.nn[0] * (a1 + (int64_t)F.nn[1] * a2) : 0;
      const bool ok = in && (!F.inst || F.inst[a] == inst_c) &&
                      !(F.fixed && F.fixed[a * F.mstride + F.moff + i]);
      const real r = rf[a * B + i];
      const real wgt = (d0 ? real(0.5) : real(1)) * (d1 ? real(0.5) : real(1)) * (d2 ? real(0.5) : real(1));
      acc = fma(wgt, ok ? r : real(0), acc);
    }
    bc[I * B + i] = acc;
  }
  if (!xc) return;
  real s = 0;
#pragma unroll
  for (int j = 0; j < B; ++j) {
    const real bj = __shfl_sync(0xffffffffu, acc, lane - i + j);
    if (live) s = fma(Cl.dinv[I * B * B + i * B + j], bj, s);
  }
  if (live) xc[I * B + i] = omega * s;
}

// (P x_c)(a) at fine node a from its 2^d candidate coarse parents: per axis
// I = a/2 (weight 1 if a is even, 1/2 if odd) and I + 1 (weight 1/2 if a is
// odd and I + 1 exists, else 0, with its index clamped).  Components i0 .. i0 + NE - 1,
// the loads (prolong_load) apart from the sum, so that a caller can issue other loads
// between them.
template <int D>
__device__ inline int64_t prolong_parent(const LevelDev &Cl, const int ac[3], int cmb, real &wgt) {
  int64_t I = 0, stride = 1;
  wgt = 1;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const int odd = ac[k] & 1, i0 = ac[k] >> 1;
    const bool up = odd && i0 + 1 < Cl.nn[k], far = (cmb >> k) & 1;
    I += stride * (far && up ? i0 + 1 : i0);
    stride *= Cl.nn[k];
    wgt = far ? (up ? wgt * real(0.5) : real(0)) : (odd ? wgt * real(0.5) : wgt);
  }
  return I;
}
template <int B, int NE, int D>
__device__ inline void prolong_load(const LevelDev &Cl, const real *__restrict__ xc, const int ac[3], int i0,
                                    real pv[1 << D][NE]) {
#pragma unroll
  for (int cmb = 0; cmb < (1 << D); ++cmb) {
    real wgt;
    const int64_t I = prolong_parent<D>(Cl, ac, cmb, wgt);
#pragma unroll
    for (int i = 0; i < NE; ++i) pv[cmb][i] = xc[I * B + i0 + i];
  }
}
template <int NE, int D>
__device__ inline void prolong_sum(const LevelDev &Cl, const int ac[3], int inst_a, const real pv[1 << D][NE],
                                   real out[NE]) {
#pragma unroll
  for (int i = 0; i < NE; ++i) out[i] = 0;
#pragma unroll
  for (int cmb = 0; cmb < (1 << D); ++cmb) {
    real w;
    const int64_t I = prolong_parent<D>(Cl, ac, cmb, w);
    if (Cl.inst && Cl.inst[I] != inst_a) w = 0;
#pragma unroll
    for (int i = 0; i < NE; ++i) out[i] = fma(w, pv[cmb][i], out[i]);
  }
}

// Window of coarse nodes that a fine row reaches: floor(a / 2) + WIN0 .. + WIN0 + W - 1
// per axis, W = 3, 4 or 5 for couplings up to 1, 2 or 3 nodes apart.  The Galerkin
// product keeps a reach of 1 at 1, and brings 2 and 3 to 2.
template <int W>
constexpr int WIN0 = W == 5 ? -2 : -1;
// whether a row of that parity reaches slot d of its window
template <int W>
__device__ __forceinline__ bool win_reaches(int a, int d) {
  return W == 3 ? !(d == -1 && (a & 1)) : W == 4 ? !(d == 2 && !(a & 1)) : true;
}

// A fine row that contributes nothing to the Galerkin product: a stencil row
// without coupling, or a finest-level row whose DOFs are all fixed (its
// transfers are masked).  On levels of VOID_ROWS rows and more k_mg_ap leaves such a
// row's T unwritten and its readers skip the row (on the slope, the grid nodes
// outside the material); on smaller ones it writes zeros, so that k_mg_post need not
// wait for the test before it loads.
constexpr int64_t VOID_ROWS = 1 << 16;
template <int B, bool FST>
__device__ inline bool row_void(const LevelDev &F, int64_t a) {
  if (FST) return F.nslot[a] == 0;
  if (!F.fixed) return false;
  for (int i = 0; i < B; ++i)
    if (!F.fixed[a * F.mstride + F.moff + i]) return false;
  return true;
}

// A level's rows are split into parts until it has POST_THREADS threads: about three
// warps for each of the chip's 608 SM quarters, so that their FP64 pipes share the work.
constexpr int64_t POST_THREADS = 1 << 16;
constexpr int POST_WARPS = 16;  // warps of a block at most

// Coarse correction and first post-smoothing sweep in one pass.  With r = b - A x
// from before the restriction and T = A P from the set-up,
//   x + P e + omega Dinv (b - A (x + P e)) = x + P e + omega Dinv (r - T e):
// a row of T holds at most 3 (even) or 4 (odd) coarse nodes per axis, 43 blocks on
// average in 3D, where a row of A holds about 110 (125 on a coarse level), and
// neither the neighbours' x nor a prolongation kernel is needed.
// A lane per row, 32 consecutive rows a warp (T is stored by rows, so every load
// of it is one line).  Where a level has few rows (SPLIT), `parts` warps share the
// rows' (z, y) window lines; their sums are joined in a tree and the rows finished a
// component a warp, since a warp's FP64 instruction holds its SM quarter's pipe for
// 64 cycles and what a small level costs is its longest warp.  What the row's end
// reads is then loaded before T (its use would hold up T's loads), and in FP32; on
// large FP64 levels, bound by the pipe (90% busy), the registers cost more than that
// gives (slope: 217 against 261 ms a step).  Where the pipe is not the bound, the loads
// of a window line go out together (finest FP32 level of a 110k-node block: 175 us in
// the compiler's order, 48 so).
// Preconditioner per step, against a prolongation kernel and a sweep over A (GB300):
// 4.2M-point slope 271 -> 209 ms, mixed 141 -> 113; 163k-point block 18.6 -> 16.7, 1M-point
// block mixed 22.9 -> 18.7; 80k-point footing 5.5 -> 5.1; steps of 64 batched columns
// 53 -> 48 ms.  On the smallest level it serves (1,681 nodes) it costs what the two
// kernels did.
template <int B, int D, bool FST, int W, bool SPLIT>
__global__ void k_mg_post(LevelDev F, LevelDev Cl, const real *__restrict__ T, const real *__restrict__ x,
                          const real *__restrict__ e, const real *__restrict__ r, real *__restrict__ out,
                          real omega, int parts) {
  pdl_enter();
  __shared__ real sm[SPLIT ? POST_WARPS : 1][B][32];
  constexpr bool EARLY = SPLIT || sizeof(real) == sizeof(float);
  constexpr int NE = SPLIT ? 1 : B;  // components a lane finishes
  constexpr int BATCH = EARLY ? W : 1;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int part = SPLIT ? wid % parts : 0, grp = SPLIT ? wid / parts : wid;
  const int64_t a = ((int64_t)blockIdx.x * ((blockDim.x >> 5) / (SPLIT ? parts : 1)) + grp) * 32 + lane;
  const bool valid = a < F.nnodes;
  const bool ends = valid && (!SPLIT || part < B);
  const int i0 = SPLIT ? part : 0;
  real te[B], rv[B], xv[NE], di[NE * B];
#pragma unroll
  for (int i = 0; i < B; ++i) te[i] = 0;
  int ac[3] = {0, 0, 0};
  bool live = valid;  // T holds the row
  real pv[1 << D][NE];
  bool fx[NE];
  auto load_end = [&]() {  // loads alone: a use of one would hold up those after it
    prolong_load<B, NE, D>(Cl, e, ac, i0, pv);
#pragma unroll
    for (int j = 0; j < B; ++j) rv[j] = r[a * B + j];
#pragma unroll
    for (int i = 0; i < NE; ++i) {
      xv[i] = x[a * B + i0 + i];
      fx[i] = F.fixed && F.fixed[a * F.mstride + F.moff + i0 + i];
#pragma unroll
      for (int j = 0; j < B; ++j) di[i * B + j] = F.dinv[a * B * B + (i0 + i) * B + j];
    }
  };
  auto sum_end = [&]() {
    real pe[NE];
    prolong_sum<NE, D>(Cl, ac, F.inst ? F.inst[a] : 0, pv, pe);
#pragma unroll
    for (int i = 0; i < NE; ++i) xv[i] += fx[i] ? real(0) : pe[i];
  };
  if (valid) {
    grid_xyz(F.nn[0], F.nn[1], (int)a, ac);
    if (F.nnodes >= VOID_ROWS) live = !row_void<B, FST>(F, a);
    if (EARLY && ends) {
      load_end();
      if (!SPLIT) sum_end();
    }
  }
  if (live) {
    constexpr int NL = D == 2 ? W : W * W;
    for (int l = part; l < NL; l += SPLIT ? parts : 1) {
      const int d1 = l % W + WIN0<W>, d2 = D == 3 ? l / W + WIN0<W> : 0;
      if (!win_reaches<W>(ac[1], d1) || (D == 3 && !win_reaches<W>(ac[2], d2))) continue;
      const int j1 = (ac[1] >> 1) + d1, j2 = D == 3 ? (ac[2] >> 1) + d2 : 0;
      if (j1 < 0 || j1 >= Cl.nn[1] || j2 < 0 || j2 >= Cl.nn[2]) continue;
      const int64_t jrow = (int64_t)Cl.nn[0] * (j1 + (int64_t)Cl.nn[1] * j2);
      const real *t0 = T + (int64_t)(l * W) * (B * B) * F.nnodes + a;
#pragma unroll
      for (int q = 0; q < W; q += BATCH) {
        real tv[BATCH][B * B], ev[BATCH][B];  // the loads of a batch go out together
#pragma unroll
        for (int u = 0; u < BATCH; ++u) {
          const int j0 = (ac[0] >> 1) + q + u + WIN0<W>;
          const bool in = j0 >= 0 && j0 < Cl.nn[0];
          const real *ej = e + (jrow + (in ? j0 : 0)) * B;
#pragma unroll
          for (int k = 0; k < B * B; ++k) tv[u][k] = __ldg(t0 + (int64_t)((q + u) * B * B + k) * F.nnodes);
#pragma unroll
          for (int j = 0; j < B; ++j) {
            const real v = __ldg(ej + j);
            ev[u][j] = in ? v : real(0);
          }
        }
#pragma unroll
        for (int u = 0; u < BATCH; ++u)
#pragma unroll
          for (int i = 0; i < B; ++i)
#pragma unroll
            for (int j = 0; j < B; ++j) te[i] = fma(tv[u][i * B + j], ev[u][j], te[i]);
      }
    }
  }
  if constexpr (SPLIT) {
#pragma unroll
    for (int i = 0; i < B; ++i) sm[wid][i][lane] = te[i];
    __syncthreads();
    for (int h = parts / 2; h >= 2; h /= 2) {
      if (part < h)
#pragma unroll
        for (int i = 0; i < B; ++i) sm[wid][i][lane] = te[i] = te[i] + sm[wid + h][i][lane];
      __syncthreads();
    }
    if (ends)
#pragma unroll
      for (int i = 0; i < B; ++i) te[i] = sm[wid - part][i][lane] + sm[wid - part + 1][i][lane];
  }
  if (!ends) return;
  if (!EARLY) load_end();
  if (!EARLY || SPLIT) sum_end();
#pragma unroll
  for (int i = 0; i < NE; ++i) {
    real s = 0;
#pragma unroll
    for (int j = 0; j < B; ++j) s = fma(di[i * B + j], rv[j] - te[j], s);
    out[a * B + i0 + i] = fma(omega, s, xv[i]);
  }
}

// ---- coarse tail of a V-cycle as one dense operator
// From the first level of at most TAIL_MAX unknowns down, a V-cycle is a chain
// of small kernels that each cost 2 to 4 us whatever their work (9 of the 45
// kernels of an application per cycle on the 80k-point footing, every one on
// the column).  That part of the cycle is a fixed linear map of its right-hand
// side, so the set-up forms its matrix T by running the cycle on the unit
// vectors (k_mg_tail_build), and an application is one product x = T b
// (k_dense_apply): the same operator, its sums in another order.  The build
// runs every column independently in shared memory, TAIL_COLS columns a block
// (a level's blocks are read once for all of them), the two hierarchies of a
// preconditioner side by side.
// TAIL_MAX: a build costs about n^2 times a row's work (0.12 ms for the 966
// unknowns of the harmonic footing's A-tail), a product n^2 FMAs (1.7 us of the
// FP64 pipes at 1024).  An application on a GB300: column 37 -> 23 us, 17 x 17
// deposit (FP32) 47 -> 19, harmonic footing 76 -> 46, 80k-point footing 139 -> 109,
// 64 batched columns 430 -> 389; with 768 the harmonic footing keeps one level more.
constexpr int TAIL_MAX = 1024;
constexpr int TAIL_COLS = 2;  // (4: one block per SM by its shared memory, 331 us for the 966 unknowns below)
constexpr int TAIL_LEVELS = 8;
constexpr int TAIL_THREADS = 512;
// Shared memory of the largest tail: three vectors per level and column, under 2
// TAIL_MAX unknowns over all levels (while a level is coarsened, every axis has
// at least 3 nodes and keeps at most 2/3 of them, so a level has at most 4/9 of the
// unknowns of the one before it).  The limit is set to this constant and not to a
// tail's own size: it belongs to the kernel, which contexts of other host threads
// launch at the same time.
constexpr size_t TAIL_SMEM_MAX = sizeof(real) * 3 * TAIL_COLS * 2 * TAIL_MAX;
static_assert(TAIL_SMEM_MAX <= 227 * 1024, "a tail's vectors fit a block's shared memory");

struct TailArgs {
  int nl;  // levels of the tail, the last one the dense coarsest level
  LevelDev L[TAIL_LEVELS];
  int st0;           // the first level is a stencil level (else the block-CSR finest level)
  const real *Ai;    // inverse of the coarsest operator
  int ncoarse, n;    // unknowns of the coarsest and of the tail's first level
  real omega;
  int nsw;
  real *T;           // n x n, row-major
};

// out = b - A x (SMOOTH: x + omega Dinv (b - A x)) for TAIL_COLS columns; vectors
// [unknown][column]; a thread per row.  The thread's row sum is in slot order.
// box (or null): x and b are zero at the rows outside it, and so is out.
template <int B, int D, bool ST, bool SMOOTH>
__device__ inline void tail_rows(const LevelDev &L, const real *x, real *out, const real *b, real omega,
                                 const int *box) {
  constexpr int NC = TAIL_COLS;
  for (int a = threadIdx.x; a < (int)L.nnodes; a += blockDim.x) {
    if (box) {
      int ac[3];
      grid_xyz(L.nn[0], L.nn[1], a, ac);
      if (ac[0] < box[0] || ac[0] > box[1] || ac[1] < box[2] || ac[1] > box[3] || ac[2] < box[4] || ac[2] > box[5]) {
#pragma unroll
        for (int i = 0; i < B * NC; ++i) out[a * B * NC + i] = 0;
        continue;
      }
    }
    real acc[B][NC];
#pragma unroll
    for (int i = 0; i < B; ++i)
#pragma unroll
      for (int c = 0; c < NC; ++c) acc[i][c] = 0;
    auto add = [&](const real *blk, int64_t nb) {
#pragma unroll
      for (int j = 0; j < B; ++j)
#pragma unroll
        for (int c = 0; c < NC; ++c) {
          const real xv = x[(nb * B + j) * NC + c];
#pragma unroll
          for (int i = 0; i < B; ++i) acc[i][c] = fma(blk[i * B + j], xv, acc[i][c]);
        }
    };
    if (!ST) {
      for (int e = L.row_ptr[a]; e < L.row_ptr[a + 1]; ++e) add(L.val + (int64_t)e * B * B, L.col[e]);
    } else if (L.nslot[a] != 0) {
      int ac[3];
      grid_xyz(L.nn[0], L.nn[1], a, ac);
      const real *base = L.sval + (int64_t)a * NS_<D>::v * B * B;
      for (int s = 0; s < NS_<D>::v; ++s) {
        const int b0 = ac[0] + s % 5 - 2, b1 = ac[1] + (s / 5) % 5 - 2, b2 = ac[2] + (D == 3 ? s / 25 - 2 : 0);
        if (b0 < 0 || b0 >= L.nn[0] || b1 < 0 || b1 >= L.nn[1] || b2 < 0 || b2 >= L.nn[2]) continue;
        real blk[B * B];  // most blocks of a coarse stencil are zero: skipped by an integer test
        unsigned long long any = 0;
#pragma unroll
        for (int e = 0; e < B * B; ++e) {
          blk[e] = base[s * B * B + e];
          any |= mag_bits(blk[e]);
        }
        if (any) add(blk, b0 + (int64_t)L.nn[0] * (b1 + (int64_t)L.nn[1] * b2));
      }
    }
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      real r[B];
#pragma unroll
      for (int i = 0; i < B; ++i) r[i] = b[(a * B + i) * NC + c] - acc[i][c];
#pragma unroll
      for (int i = 0; i < B; ++i) {
        if (!SMOOTH) {
          out[(a * B + i) * NC + c] = r[i];
          continue;
        }
        real sv = 0;
#pragma unroll
        for (int j = 0; j < B; ++j) sv = fma(L.dinv[(int64_t)a * B * B + i * B + j], r[j], sv);
        out[(a * B + i) * NC + c] = x[(a * B + i) * NC + c] + omega * sv;
      }
    }
  }
}

template <int B, int D, bool SMOOTH>
__device__ inline void tail_level(const TailArgs &A, int l, const real *x, real *out, const real *b,
                                  const int *box = nullptr) {
  if (l == 0 && !A.st0) tail_rows<B, D, false, SMOOTH>(A.L[l], x, out, b, A.omega, box);
  else tail_rows<B, D, true, SMOOTH>(A.L[l], x, out, b, A.omega, box);
}

// Columns c0 .. c0 + TAIL_COLS - 1 of T.  Dynamic shared memory: per level x,
// b and r (x of the next sweep), tail_smem() bytes.
template <int B, int D>
__device__ void tail_build(const TailArgs &A, int c0, real *sm) {
  constexpr int NC = TAIL_COLS;
  real *x[TAIL_LEVELS], *b[TAIL_LEVELS], *r[TAIL_LEVELS];
  for (int l = 0; l < A.nl; ++l) {
    const int64_t n = A.L[l].nnodes * B * NC;
    x[l] = sm;
    b[l] = sm + n;
    r[l] = sm + 2 * n;
    sm += 3 * n;
  }
  for (int t = threadIdx.x; t < A.n * NC; t += blockDim.x) b[0][t] = t / NC == c0 + t % NC ? real(1) : real(0);
  __syncthreads();
  auto swap = [](real *&p, real *&q) {
    real *t = p;
    p = q;
    q = t;
  };
  for (int l = 0; l + 1 < A.nl; ++l) {
    const LevelDev &L = A.L[l], &Ln = A.L[l + 1];
    // first sweep from zero: x = omega Dinv b
    for (int t = threadIdx.x; t < (int)L.nnodes * B * NC; t += blockDim.x) {
      const int c = t % NC, a = t / NC / B, i = t / NC % B;
      real sv = 0;
      for (int j = 0; j < B; ++j) sv = fma(L.dinv[(int64_t)a * B * B + i * B + j], b[l][(a * B + j) * NC + c], sv);
      x[l][t] = A.omega * sv;
    }
    __syncthreads();
    for (int k = 1; k < A.nsw; ++k) {
      tail_level<B, D, true>(A, l, x[l], r[l], b[l]);
      __syncthreads();
      swap(x[l], r[l]);
    }
    // the first residual of the unit vectors is zero beyond their nodes' stencils
    int box[6];
    const bool near = l == 0 && A.nsw == 1;
    if (near) {
      int p[3], q[3];
      grid_xyz(L.nn[0], L.nn[1], c0 / B, p);
      grid_xyz(L.nn[0], L.nn[1], min(c0 + NC - 1, A.n - 1) / B, q);
      const int reach = A.st0 ? 2 : 3;
      if (p[1] != q[1] || p[2] != q[2]) {  // the columns' nodes run over a row's end
        p[0] = 0;
        q[0] = L.nn[0] - 1;
      }
      if (p[2] != q[2]) {
        p[1] = 0;
        q[1] = L.nn[1] - 1;
      }
      for (int k = 0; k < 3; ++k) {
        box[2 * k] = min(p[k], q[k]) - reach;
        box[2 * k + 1] = max(p[k], q[k]) + reach;
      }
    }
    tail_level<B, D, false>(A, l, x[l], r[l], b[l], near ? box : nullptr);
    __syncthreads();
    for (int t = threadIdx.x; t < (int)Ln.nnodes * B * NC; t += blockDim.x) {  // restriction
      const int c = t % NC, I = t / NC / B, i = t / NC % B;
      int Ic[3];
      grid_xyz(Ln.nn[0], Ln.nn[1], I, Ic);
      real acc = 0;
      const int lo2 = D == 3 ? -1 : 0, hi2 = D == 3 ? 1 : 0;
      for (int d2 = lo2; d2 <= hi2; ++d2)
        for (int d1 = -1; d1 <= 1; ++d1)
          for (int d0 = -1; d0 <= 1; ++d0) {
            const int a0 = 2 * Ic[0] + d0, a1 = 2 * Ic[1] + d1, a2 = D == 3 ? 2 * Ic[2] + d2 : 0;
            if (a0 < 0 || a0 >= L.nn[0] || a1 < 0 || a1 >= L.nn[1] || a2 < 0 || a2 >= L.nn[2]) continue;
            const int64_t a = a0 + (int64_t)L.nn[0] * (a1 + (int64_t)L.nn[1] * a2);
            if (L.inst && L.inst[a] != Ln.inst[I]) continue;
            const real wgt = pw(a0, Ic[0]) * pw(a1, Ic[1]) * (D == 3 ? pw(a2, Ic[2]) : real(1));
            acc += wgt * free_w(L, a, i) * r[l][(a * B + i) * NC + c];
          }
      b[l + 1][t] = acc;
    }
    __syncthreads();
  }
  {  // exact solve on the coarsest grid
    const int lc = A.nl - 1;
    for (int t = threadIdx.x; t < A.ncoarse * NC; t += blockDim.x) {
      const int c = t % NC, i = t / NC;
      real sv = 0;
      for (int j = 0; j < A.ncoarse; ++j) sv = fma(A.Ai[(int64_t)i * A.ncoarse + j], b[lc][j * NC + c], sv);
      x[lc][t] = sv;
    }
    __syncthreads();
  }
  for (int l = A.nl - 2; l >= 0; --l) {
    const LevelDev &L = A.L[l], &Ln = A.L[l + 1];
    for (int t = threadIdx.x; t < (int)L.nnodes * B * NC; t += blockDim.x) {  // prolongation
      const int c = t % NC, a = t / NC / B, i = t / NC % B;
      int ac[3];
      grid_xyz(L.nn[0], L.nn[1], a, ac);
      const int inst_a = L.inst ? L.inst[a] : 0;
      real acc = 0;
      for (int cmb = 0; cmb < (1 << D); ++cmb) {
        real w = 1;
        int I[3] = {0, 0, 0};
        for (int k = 0; k < D; ++k) {
          const int odd = ac[k] & 1, up = (cmb >> k) & 1;
          I[k] = (ac[k] >> 1) + up;
          w *= up ? (odd && I[k] < Ln.nn[k] ? real(0.5) : real(0)) : (odd ? real(0.5) : real(1));
        }
        if (w == real(0)) continue;
        const int64_t In = I[0] + (int64_t)Ln.nn[0] * (I[1] + (int64_t)Ln.nn[1] * I[2]);
        if (Ln.inst && Ln.inst[In] != inst_a) continue;
        acc = fma(w, x[l + 1][(In * B + i) * NC + c], acc);
      }
      x[l][t] += free_w(L, a, i) * acc;
    }
    __syncthreads();
    for (int k = 0; k < A.nsw; ++k) {
      tail_level<B, D, true>(A, l, x[l], r[l], b[l]);
      __syncthreads();
      swap(x[l], r[l]);
    }
  }
  for (int t = threadIdx.x; t < A.n * NC; t += blockDim.x) {
    const int c = c0 + t % NC;
    if (c < A.n) A.T[(int64_t)(t / NC) * A.n + c] = x[0][t];
  }
}

// blocks 0 .. nblk0 - 1: the A hierarchy (B = D), the others the S hierarchy
template <int D>
__global__ void __launch_bounds__(TAIL_THREADS) k_mg_tail_build(TailArgs A, TailArgs S, int nblk0) {
  extern __shared__ __align__(16) unsigned char dyn_smem[];
  real *sm = reinterpret_cast<real *>(dyn_smem);
  if ((int)blockIdx.x < nblk0) tail_build<D, D>(A, blockIdx.x * TAIL_COLS, sm);
  else tail_build<1, D>(S, ((int)blockIdx.x - nblk0) * TAIL_COLS, sm);
}

// Galerkin product P^T A P in two passes, from the block-CSR finest level
// (couplings up to 3 apart per axis) or a stencil level (up to 2 apart):
//   k_mg_ap:   T_a(J) = sum_b w_bJ A_ab over the children b of J, for every
//              fine row a and coarse node J of the W^d window of the coarse
//              nodes a row can reach (WIN0); thread per (window slot, a).  T is
//              kept: k_mg_post applies it;
//   k_mg_rap2: A_c(I, J) = sum_a w_aI T_a(J) over the 3^d children a of I;
//              thread per (stencil slot, I).
// Dirichlet DOFs are masked out of the finest level's transfers only, and
// instances are kept apart on every level; grouped as (P^T (A P)), a coarse
// entry costs a few lookups and 3^d FMA blocks instead of one per (a, b) pair
// (measured on the slope's stencil levels: the one-pass product took 20 ms
// per set-up).
template <int B, int D, bool FST, int W>
__global__ void k_mg_ap(LevelDev F, LevelDev Cl, real *__restrict__ T) {
  constexpr int NS = D == 2 ? W * W : W * W * W;  // window slots
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // the lanes of a warp take one window slot of consecutive fine rows (the same
  // loop bounds up to the parity of a), and T is stored [slot][value][row] so
  // that their results are written side by side; a tile of AP_ROWS rows takes all
  // its slots before the next one, so that the row's blocks are read from DRAM
  // once and not once per slot that reaches them (the set-up class of the
  // 4.2M-point slope, with the split in one pass and the fixed-stress gather:
  // 46.8 -> 35.2 ms in FP64, 29.1 -> 20.1 ms a set-up in FP32)
  const int64_t tile = t / (AP_ROWS * NS);
  const int rem = (int)(t - tile * (AP_ROWS * NS));
  const int64_t a = tile * AP_ROWS + rem % AP_ROWS;
  const int s = rem / AP_ROWS;
  if (a >= F.nnodes) return;
  const bool none = row_void<B, FST>(F, a);
  if (none && F.nnodes >= VOID_ROWS) return;
  int fa[3], Jc[3];
  grid_xyz(F.nn[0], F.nn[1], (int)a, fa);
  Jc[0] = (fa[0] >> 1) + s % W + WIN0<W>;
  Jc[1] = (fa[1] >> 1) + (s / W) % W + WIN0<W>;
  Jc[2] = D == 3 ? (fa[2] >> 1) + s / (W * W) + WIN0<W> : 0;
  real acc[B * B];
  for (int i = 0; i < B * B; ++i) acc[i] = 0.0;
  if (!none && Jc[0] >= 0 && Jc[0] < Cl.nn[0] && Jc[1] >= 0 && Jc[1] < Cl.nn[1] && Jc[2] >= 0 && Jc[2] < Cl.nn[2]) {
    const int64_t Jn = Jc[0] + (int64_t)Cl.nn[0] * (Jc[1] + (int64_t)Cl.nn[1] * Jc[2]);
    int blo[3], bhi[3];  // children of J within reach of a (and inside the grid)
    for (int k = 0; k < 3; ++k) {
      const int lo = 2 * Jc[k] - 1 > fa[k] - 3 ? 2 * Jc[k] - 1 : fa[k] - 3;
      const int hi = 2 * Jc[k] + 1 < fa[k] + 3 ? 2 * Jc[k] + 1 : fa[k] + 3;
      blo[k] = lo > 0 ? lo : 0;
      bhi[k] = hi < F.nn[k] - 1 ? hi : F.nn[k] - 1;
    }
    if (D == 2) blo[2] = bhi[2] = 0;
    for (int b2 = blo[2]; b2 <= bhi[2]; ++b2)
      for (int b1 = blo[1]; b1 <= bhi[1]; ++b1)
        for (int b0 = blo[0]; b0 <= bhi[0]; ++b0) {
          const int64_t b = b0 + (int64_t)F.nn[0] * (b1 + (int64_t)F.nn[1] * b2);
          if (F.inst && F.inst[b] != Cl.inst[Jn]) continue;
          const real *blk;
          if (!FST) {  // finest level: block-CSR, found by the coupling mask
            const int e = mask_block<D>(F.mask, F.row_ptr, (int)a, b0 - fa[0], b1 - fa[1], b2 - fa[2]);
            if (e < 0) continue;
            blk = F.val + (int64_t)e * B * B;
          } else {     // stencil level: the 5^d slot of b - a
            const int d0 = b0 - fa[0], d1 = b1 - fa[1], d2 = b2 - fa[2];
            if (d0 < -2 || d0 > 2 || d1 < -2 || d1 > 2 || d2 < -2 || d2 > 2) continue;
            blk = F.sval + (a * NS_<D>::v + (d0 + 2) + 5 * (d1 + 2) + (D == 3 ? 25 * (d2 + 2) : 0)) * B * B;
          }
          const real w = pw(b0, Jc[0]) * pw(b1, Jc[1]) * (D == 3 ? pw(b2, Jc[2]) : 1.0);
          for (int j = 0; j < B; ++j) {
            const real wj = FST ? w : w * free_w(F, b, j);  // Dirichlet masks: finest transfers only
            for (int i = 0; i < B; ++i) acc[i * B + j] = fma(wj, blk[i * B + j], acc[i * B + j]);
          }
        }
  }
  for (int i = 0; i < B * B; ++i) T[((int64_t)s * (B * B) + i) * F.nnodes + a] = acc[i];
}

template <int B, int D, bool FST, int W>
__global__ void k_mg_rap2(LevelDev F, LevelDev Cl, const real *__restrict__ T) {
  constexpr int NS = NS_<D>::v;
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  // mapped as k_mg_ap: the lanes take consecutive coarse nodes I of one stencil
  // slot, so a child a = 2 I + d of every lane reads the same window slot of T at
  // every other fine row
  const int64_t tile = t / (AP_ROWS * NS);
  const int rem = (int)(t - tile * (AP_ROWS * NS));
  const int64_t I = tile * AP_ROWS + rem % AP_ROWS;
  const int s = rem / AP_ROWS;
  if (I >= Cl.nnodes) return;
  int Ic[3], Jc[3];
  grid_xyz(Cl.nn[0], Cl.nn[1], (int)I, Ic);
  Jc[0] = Ic[0] + s % 5 - 2;
  Jc[1] = Ic[1] + (s / 5) % 5 - 2;
  Jc[2] = D == 3 ? Ic[2] + s / 25 - 2 : 0;
  real acc[B * B];
  for (int i = 0; i < B * B; ++i) acc[i] = 0.0;
  if (Jc[0] >= 0 && Jc[0] < Cl.nn[0] && Jc[1] >= 0 && Jc[1] < Cl.nn[1] && Jc[2] >= 0 && Jc[2] < Cl.nn[2]) {
    const int lo2 = D == 3 ? -1 : 0, hi2 = D == 3 ? 1 : 0;
    for (int a2 = lo2; a2 <= hi2; ++a2)
      for (int a1 = -1; a1 <= 1; ++a1)
        for (int a0 = -1; a0 <= 1; ++a0) {
          const int fa[3] = {2 * Ic[0] + a0, 2 * Ic[1] + a1, D == 3 ? 2 * Ic[2] + a2 : 0};
          if (fa[0] < 0 || fa[0] >= F.nn[0] || fa[1] < 0 || fa[1] >= F.nn[1] || fa[2] < 0 || fa[2] >= F.nn[2])
            continue;
          // slot of J in a's window; outside it, T_a(J) is zero (J out of reach)
          const int d0 = Jc[0] - (fa[0] >> 1), d1 = Jc[1] - (fa[1] >> 1), d2 = D == 3 ? Jc[2] - (fa[2] >> 1) : 0;
          constexpr int lo = WIN0<W>, hi = lo + W - 1;
          if (d0 < lo || d0 > hi || d1 < lo || d1 > hi || (D == 3 && (d2 < lo || d2 > hi))) continue;
          const int64_t a = fa[0] + (int64_t)F.nn[0] * (fa[1] + (int64_t)F.nn[1] * fa[2]);
          if (F.inst && F.inst[a] != Cl.inst[I]) continue;
          const real wa = pw(fa[0], Ic[0]) * pw(fa[1], Ic[1]) * (D == 3 ? pw(fa[2], Ic[2]) : 1.0);
          real wi[B];
          bool any = false;
          for (int i = 0; i < B; ++i) {
            wi[i] = FST ? wa : wa * free_w(F, a, i);
            any |= wi[i] != real(0);
          }
          // a row without contribution (row_void): T_a was not written
          if (FST ? F.nslot[a] == 0 : !any) continue;
          const int sl = (d0 - lo) + W * (d1 - lo) + (D == 3 ? W * W * (d2 - lo) : 0);
          const real *ta = T + (int64_t)sl * (B * B) * F.nnodes + a;
          for (int i = 0; i < B; ++i)
            for (int j = 0; j < B; ++j)
              acc[i * B + j] = fma(wi[i], ta[(int64_t)(i * B + j) * F.nnodes], acc[i * B + j]);
        }
  }
  for (int i = 0; i < B * B; ++i) Cl.sval[(I * NS + s) * B * B + i] = acc[i];
}

// Nonzero blocks of each coarse row (a block is zero when the product never
// reached it: the coupling is absent), so that the row kernels skip the rows
// of nodes without coupling.  A warp per row (a thread per row read its up to 9 KB
// alone: 110 us on a 3,000-node level).
template <int B, int D>
__global__ void k_mg_rowcount(LevelDev Cl) {
  constexpr int NS = NS_<D>::v;
  const int64_t I = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (I >= Cl.nnodes) return;
  const real *row = Cl.sval + I * NS * B * B;
  int cnt = 0;
  for (int s0 = 0; s0 < NS; s0 += 32) {
    const int s = s0 + lane;
    bool nz = false;
    if (s < NS)
#pragma unroll
      for (int e = 0; e < B * B; ++e) nz |= row[s * B * B + e] != real(0);
    cnt += __popc(__ballot_sync(0xffffffffu, nz));
  }
  if (lane == 0) Cl.nslot[I] = (uint8_t)cnt;
}

}  // namespace MG_NS

// ============================================================== hierarchy
template <>
struct MGHier<MG_REAL> {
  int B = 1, nlev = 0;
  MG_NS::LevelDev L[16];
  MG_REAL *x[16], *x2[16], *b[16], *r[16];
  // dense coarsest operator (LU factors after set-up), its inverse, the factors' transpose
  MG_REAL *Ad = nullptr, *Ai = nullptr, *At = nullptr;
  int *piv = nullptr;                    // row interchanges of the LU factorisation
  MG_REAL *ap[16] = {};                  // A P of a level and the next one, on its window (k_mg_ap)
  int win = 4, cwin = 4;                 // windows of the finest level and of the coarse levels
  int ap_slots = 0;                      // window slots ap[0] has room for
  int ncoarse = 0;                       // unknowns of the coarsest level
  int tail = 15;                         // first level of the dense tail (nlev - 1: the coarsest alone)
  MG_REAL *T = nullptr;                  // its operator
};

namespace MG_NS {

// f(W) with the compile-time window
template <typename F>
inline void with_window(int win, F &&f) {
  if (win == 3) f(std::integral_constant<int, 3>{});
  else if (win == 5) f(std::integral_constant<int, 5>{});
  else f(std::integral_constant<int, 4>{});
}

template <int B, int D>
void mg_setup_t(Ctx &c, MGHier<real> &H) {
  for (int l = 0; l < H.nlev; ++l) {
    LevelDev &L = H.L[l];
    const int nbk = nblk(L.nnodes);
    if (l > 0) {
      constexpr int NS = NS_<D>::v;
      const int g2 = nblk(ap_threads(L.nnodes, NS));
      const int64_t nf = H.L[l - 1].nnodes;
      real *T = H.ap[l - 1];
      with_window(l == 1 ? H.win : H.cwin, [&](auto win) {
        constexpr int W = decltype(win)::value, N = D == 2 ? W * W : W * W * W;
        if (l == 1) {
          k_mg_ap<B, D, false, W><<<nblk(ap_threads(nf, N)), TPB, 0, c.st>>>(H.L[0], L, T);
          k_mg_rap2<B, D, false, W><<<g2, TPB, 0, c.st>>>(H.L[0], L, T);
        } else if constexpr (W < 5) {
          k_mg_ap<B, D, true, W><<<nblk(ap_threads(nf, N)), TPB, 0, c.st>>>(H.L[l - 1], L, T);
          k_mg_rap2<B, D, true, W><<<g2, TPB, 0, c.st>>>(H.L[l - 1], L, T);
        }
      });
      k_mg_rowcount<B, D><<<nblk(L.nnodes * 32), TPB, 0, c.st>>>(L);
      UPMPM_LAUNCH(c);
      UPMPM_LAUNCH(c);
      UPMPM_LAUNCH(c);
      k_mg_dinv<B, D, true><<<nbk, TPB, 0, c.st>>>(L, c.err);
    } else {
      k_mg_dinv<B, D, false><<<nbk, TPB, 0, c.st>>>(L, c.err);
    }
    UPMPM_LAUNCH(c);
  }
  // coarsest level: dense inverse
  LevelDev &Lc = H.L[H.nlev - 1];
  const int64_t n = H.ncoarse;
  if (H.nlev == 1) k_dense_fill<B, D, false><<<nblk(n * n), TPB, 0, c.st>>>(Lc, H.Ad);
  else k_dense_fill<B, D, true><<<nblk(n * n), TPB, 0, c.st>>>(Lc, H.Ad);
  UPMPM_LAUNCH(c);
}

// Inverses of the coarsest operators of two hierarchies, in one launch.
void dense_invert_pair(Ctx &c, MGHier<real> &H0, MGHier<real> &H1) {
  const int nmax = H0.ncoarse > H1.ncoarse ? H0.ncoarse : H1.ncoarse;
  int ns = nmax;
  while (sizeof(real) * (size_t)ns * (ns | 1) > DENSE_SMEM_MAX) --ns;
  const size_t bytes = sizeof(real) * (size_t)ns * (ns | 1);
  cudaFuncSetAttribute(k_dense_lu, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DENSE_SMEM_MAX);
  const DenseJob a{H0.ncoarse, H0.Ad, H0.Ai, H0.At, H0.piv}, b{H1.ncoarse, H1.Ad, H1.Ai, H1.At, H1.piv};
  k_dense_lu<<<2, DENSE_LU_THREADS, bytes, c.st>>>(a, b, ns);
  k_dense_inv_cols<<<dim3(nblk(nmax, 4), 2), 128, 0, c.st>>>(a, b);
  c.launches += 2;
}

real mg_omega(const Ctx &c);

// Dense tail operators of the two hierarchies (after the coarsest inverses).
// finest_only: the coarse levels are those of an earlier set-up, so only a tail
// that starts at the finest level has changed.
void tail_build_pair(Ctx &c, MGHier<real> &HA, MGHier<real> &HS, bool finest_only) {
  auto args = [&](MGHier<real> &H, size_t *smem) {
    TailArgs A{};
    if (H.tail == H.nlev - 1 || (finest_only && H.tail > 0)) return A;
    A.nl = H.nlev - H.tail;
    int64_t vals = 0;
    for (int l = 0; l < A.nl; ++l) {
      A.L[l] = H.L[H.tail + l];
      vals += 3 * A.L[l].nnodes * H.B * TAIL_COLS;
    }
    A.st0 = H.tail > 0;
    A.Ai = H.Ai;
    A.ncoarse = H.ncoarse;
    A.n = (int)(A.L[0].nnodes * H.B);
    A.omega = mg_omega(c);
    A.nsw = c.mg_sweeps();
    A.T = H.T;
    *smem = std::max(*smem, sizeof(real) * (size_t)vals);
    return A;
  };
  size_t smem = 0;
  const TailArgs A = args(HA, &smem), S = args(HS, &smem);
  const int na = nblk(A.n, TAIL_COLS), ns = nblk(S.n, TAIL_COLS);
  if (na + ns == 0) return;
  auto build = [&](auto kernel) {
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TAIL_SMEM_MAX);
    kernel<<<na + ns, TAIL_THREADS, smem, c.st>>>(A, S, na);
  };
  if (c.d == 2) build(k_mg_tail_build<2>);
  else build(k_mg_tail_build<3>);
  UPMPM_LAUNCH(c);
}

// Damping of the block-Jacobi smoother.  A damped Jacobi sweep is stable only
// while omega * lambda_max(Dinv A) < 2 on every level.  Measured lambda_max:
// at most 2.5 for the plane-strain blocks of the strip footing (2D), 3.25 on
// the 3D consolidation block and 3.5 next to the inclined free surface of the
// 3D slope, where 0.6 made the V(2,2)-cycle diverge (FGMRES at its cap; 14
// iterations instead of 232 with 0.5 on a 32 x 32 x 16 slope).  The default
// cycle is V(1,1) (0.7 in 2D, 0.5 in 3D): on the full-size slope it took
// fewer FGMRES iterations than V(2,2) at 0.56 of its cost per application,
// and V(3,3) stalled there.
// (the defaults of Ctx::mg_omega; mpm_options.mg_omega overrides them)
real mg_omega(const Ctx &c) { return (real)c.mg_omega(); }

// one damped block-Jacobi sweep on level l: x <- x + omega Dinv (b - A x)
template <int B, int D>
void sweep(Ctx &c, MGHier<real> &H, int l) {
  LevelDev &L = H.L[l];
  if (l == 0 && B <= 2) {
    constexpr int SPL = B <= 2 ? 4 / B : 1;
    const Geom g = geom(c, L.nnodes * B * SPL);
    launch_pdl(c, k_mg_csr_row<B, SPL, true>, g.blocks, g.tpb, 0, L, (const real *)H.x[l], H.x2[l],
               (const real *)H.b[l], mg_omega(c));
  } else {
    with_lanes<D>(L.nnodes, [&](auto lanes) {
      constexpr int LN = decltype(lanes)::value;
      const Geom g = geom(c, L.nnodes * LN);
      auto go = [&](auto kernel) {
        launch_pdl(c, kernel, g.blocks, g.tpb, 0, L, (const real *)H.x[l], H.x2[l], (const real *)H.b[l],
                   mg_omega(c), 0);
      };
      if (l == 0) go(k_mg_smooth<B, D, false, LN>);
      else go(k_mg_smooth<B, D, true, LN>);
    });
  }
  std::swap(H.x[l], H.x2[l]);
}

// V(k,k)-cycle on level l (k = c.mg_sweeps(), default 1).  On entry b[l]
// holds the rhs and x[l] the first pre-smoothing sweep from zero (omega Dinv
// b, pointwise), done by the kernel that produced b[l]; on return x[l] holds
// the result.
template <int B, int D>
void vcycle_t(Ctx &c, MGHier<real> &H, int l) {
  if (l == H.tail) {  // the rest of the cycle (the exact solve on the coarsest grid)
    const bool last = l == H.nlev - 1;
    const int n = (int)(H.L[l].nnodes * B);
    const Geom g = geom(c, (int64_t)n * 32);
    launch_pdl(c, k_dense_apply, g.blocks, g.tpb, 0, n, (const real *)(last ? H.Ai : H.T), (const real *)H.b[l],
               H.x[l]);
    return;
  }
  LevelDev &L = H.L[l], &Ln = H.L[l + 1];
  real *xn_first = l + 1 == H.tail ? nullptr : H.x[l + 1];
  for (int k = 1; k < c.mg_sweeps(); ++k) sweep<B, D>(c, H, l);  // pre-smoothing after the first
  const Geom gc = geom(c, (Ln.nnodes + restrict_nodes<B>() - 1) / restrict_nodes<B>() * 32);
  if (l == 0 && B <= 2) {
    constexpr int SPL = B <= 2 ? 4 / B : 1;
    const Geom g0 = geom(c, L.nnodes * B * SPL);
    launch_pdl(c, k_mg_csr_row<B, SPL, false>, g0.blocks, g0.tpb, 0, L, (const real *)H.x[l], H.r[l],
               (const real *)H.b[l], mg_omega(c));
  } else {
    with_lanes<D>(L.nnodes, [&](auto lanes) {
      constexpr int LN = decltype(lanes)::value;
      const Geom g = geom(c, L.nnodes * LN);
      auto go = [&](auto kernel) {
        launch_pdl(c, kernel, g.blocks, g.tpb, 0, L, (const real *)H.x[l], (const real *)H.b[l], H.r[l]);
      };
      if (l == 0) go(k_mg_resid<B, D, false, LN>);
      else go(k_mg_resid<B, D, true, LN>);
    });
  }
  launch_pdl(c, k_mg_restrict<B, D>, gc.blocks, gc.tpb, 0, L, Ln, (const real *)H.r[l], H.b[l + 1], xn_first,
             mg_omega(c));
  vcycle_t<B, D>(c, H, l + 1);
  // coarse correction and first post-smoothing sweep
  int parts = 1;
  while (parts < (D == 2 ? 4 : 16) && L.nnodes * parts < POST_THREADS) parts *= parts == 1 ? D + D - 2 : 2;
  const int warps = parts < 4 ? 4 : parts, rows = warps / parts * 32;
  auto post = [&](auto kernel) {
    launch_pdl(c, kernel, nblk(L.nnodes, rows), 32 * warps, 0, L, Ln, (const real *)H.ap[l], (const real *)H.x[l],
               (const real *)H.x[l + 1], (const real *)H.r[l], H.x2[l], mg_omega(c), parts);
  };
  with_window(l == 0 ? H.win : H.cwin, [&](auto win) {
    constexpr int W = decltype(win)::value;
    if (l == 0) parts > 1 ? post(k_mg_post<B, D, false, W, true>) : post(k_mg_post<B, D, false, W, false>);
    else if constexpr (W < 5) parts > 1 ? post(k_mg_post<B, D, true, W, true>) : post(k_mg_post<B, D, true, W, false>);
  });
  std::swap(H.x[l], H.x2[l]);
  for (int k = 1; k < c.mg_sweeps(); ++k) sweep<B, D>(c, H, l);  // post-smoothing sweeps after it
}

// Allocate a hierarchy for block size B over the grid's node lattice; level 0
// refers to a block-CSR operator given at setup.
int mg_alloc(Ctx &c, MGHier<real> &H, int B) {
  H.B = B;
  const int D = c.d;
  const int NS = D == 2 ? 25 : 125;
  int nn[3] = {c.g.nn[0], c.g.nn[1], c.g.nn[2]};
  // instance of every node of the current level (host); level l + 1 takes
  // the instance of the fine node at the same place (2I)
  std::vector<int32_t> imap((size_t)nn[0] * nn[1] * nn[2], -1), inext;
  for (size_t i = 0; i < c.inst_h.size(); ++i) {
    const InstDev &I = c.inst_h[i];
    const int64_t m0 = I.nc[0] + 1, m1 = D > 1 ? I.nc[1] + 1 : 1, m2 = D > 2 ? I.nc[2] + 1 : 1;
    for (int64_t t = 0; t < m0 * m1 * m2; ++t) {
      const int64_t i0 = t % m0, i1 = (t / m0) % m1, i2 = t / (m0 * m1);
      imap[(i0 + I.off[0]) + (int64_t)nn[0] * ((i1 + I.off[1]) + (int64_t)nn[1] * (i2 + I.off[2]))] = (int32_t)i;
    }
  }
  int l = 0;
  while (true) {
    LevelDev &L = H.L[l];
    for (int k = 0; k < 3; ++k) L.nn[k] = nn[k];
    L.nnodes = (int64_t)nn[0] * nn[1] * nn[2];
    L.row_ptr = nullptr;
    L.col = nullptr;
    L.val = nullptr;
    L.sval = nullptr;
    L.nslot = nullptr;
    L.fixed = nullptr;
    L.mask = nullptr;
    L.mstride = 1;
    L.moff = 0;
    const int64_t vb = L.nnodes * B;
    if (cudaMalloc(&L.dinv, sizeof(real) * L.nnodes * B * B) ||
        cudaMalloc(&H.x[l], sizeof(real) * vb) || cudaMalloc(&H.x2[l], sizeof(real) * vb) ||
        cudaMalloc(&H.b[l], sizeof(real) * vb) || cudaMalloc(&H.r[l], sizeof(real) * vb))
      return MPM_ERR_NO_MEMORY;
    if (l > 0 && (cudaMalloc(&L.sval, sizeof(real) * L.nnodes * NS * B * B) || cudaMalloc(&L.nslot, L.nnodes)))
      return MPM_ERR_NO_MEMORY;
    int32_t *dinst = nullptr;
    if (c.ninst > 1) {
      if (cudaMalloc(&dinst, sizeof(int32_t) * L.nnodes) != cudaSuccess) return MPM_ERR_NO_MEMORY;
      cudaMemcpy(dinst, imap.data(), sizeof(int32_t) * L.nnodes, cudaMemcpyHostToDevice);
    }
    L.inst = dinst;
    ++l;
    int mn = 1 << 30;
    for (int k = 0; k < D; ++k) mn = nn[k] < mn ? nn[k] : mn;
    // the coarsest level is solved exactly: stop at <= 64 nodes or a 2-node axis
    if (mn <= 2 || L.nnodes <= 64 || l >= 15) break;
    int nc[3] = {nn[0], nn[1], nn[2]};
    for (int k = 0; k < D; ++k) nc[k] = (nn[k] + 1) / 2;
    inext.assign((size_t)nc[0] * nc[1] * nc[2], -1);
    for (int64_t I2 = 0; I2 < nc[2]; ++I2)
      for (int64_t I1 = 0; I1 < nc[1]; ++I1)
        for (int64_t I0 = 0; I0 < nc[0]; ++I0) {
          const int64_t f0 = 2 * I0, f1 = D > 1 ? 2 * I1 : I1, f2 = D > 2 ? 2 * I2 : I2;
          inext[I0 + nc[0] * (I1 + nc[1] * I2)] = imap[f0 + nn[0] * (f1 + nn[1] * f2)];
        }
    imap.swap(inext);
    for (int k = 0; k < 3; ++k) nn[k] = nc[k];
  }
  H.nlev = l;
  H.ncoarse = (int)(H.L[l - 1].nnodes * B);
  if (H.ncoarse > 1024) {  // an axis of 2 nodes stops the coarsening early (a thin grid)
    c.last_error = "multigrid: the coarsest level has more than 1024 unknowns (one grid axis of very few "
                   "cells against a long one)";
    return MPM_ERR_BAD_ARG;
  }
  if (cudaMalloc(&H.Ad, sizeof(real) * H.ncoarse * H.ncoarse) ||
      cudaMalloc(&H.Ai, sizeof(real) * H.ncoarse * H.ncoarse) ||
      cudaMalloc(&H.At, sizeof(real) * H.ncoarse * H.ncoarse) || cudaMalloc(&H.piv, 2 * sizeof(int) * H.ncoarse))
    return MPM_ERR_NO_MEMORY;
  H.tail = H.nlev - 1;
  while (H.tail > 0 && H.L[H.tail - 1].nnodes * B <= TAIL_MAX && H.nlev - H.tail < TAIL_LEVELS) --H.tail;
  if (H.tail < H.nlev - 1) {
    const int64_t n = H.L[H.tail].nnodes * B;
    if (cudaMalloc(&H.T, sizeof(real) * n * n)) return MPM_ERR_NO_MEMORY;
  }
  H.ap_slots = D == 2 ? 16 : 64;
  for (int k = 0; k + 1 < H.nlev; ++k)
    if (cudaMalloc(&H.ap[k], sizeof(real) * H.L[k].nnodes * H.ap_slots * B * B)) return MPM_ERR_NO_MEMORY;
  return MPM_OK;
}

void mg_free(MGHier<real> &H) {
  cudaFree(H.Ad);
  cudaFree(H.Ai);
  cudaFree(H.At);
  cudaFree(H.piv);
  for (real *&p : H.ap) {
    cudaFree(p);
    p = nullptr;
  }
  cudaFree(H.T);
  H.Ad = H.Ai = H.At = H.T = nullptr;
  H.piv = nullptr;
  for (int l = 0; l < H.nlev; ++l) {
    cudaFree(const_cast<int32_t *>(H.L[l].inst));
    H.L[l].inst = nullptr;
    cudaFree(H.L[l].dinv);
    cudaFree(H.L[l].sval);
    cudaFree(H.L[l].nslot);
    cudaFree(H.x[l]);
    cudaFree(H.x2[l]);
    cudaFree(H.b[l]);
    cudaFree(H.r[l]);
  }
  H.nlev = 0;
}

// The finest level's block-Jacobi inverses and A P only: the coarse levels keep the
// Galerkin product of an earlier set-up (mpm_options.precond_reuse).
template <int B, int D>
void mg_refresh_t(Ctx &c, MGHier<real> &H) {
  if (H.nlev > 1) {
    const int64_t nf = H.L[0].nnodes;
    with_window(H.win, [&](auto win) {
      constexpr int W = decltype(win)::value, N = D == 2 ? W * W : W * W * W;
      k_mg_ap<B, D, false, W><<<nblk(ap_threads(nf, N)), TPB, 0, c.st>>>(H.L[0], H.L[1], H.ap[0]);
    });
    UPMPM_LAUNCH(c);
  }
  k_mg_dinv<B, D, false><<<nblk(H.L[0].nnodes), TPB, 0, c.st>>>(H.L[0], c.err);
  UPMPM_LAUNCH(c);
}

void mg_setup(Ctx &c, MGHier<real> &H, const int32_t *row_ptr, const int32_t *col, const real *val,
              int moff, bool coarse) {
  H.L[0].row_ptr = row_ptr;
  H.L[0].col = col;
  H.L[0].val = val;
  H.L[0].fixed = c.fixed;
  H.L[0].mstride = c.nb;
  H.L[0].moff = moff;
  H.L[0].mask = c.row_mask;
  if (c.d == 2) {
    if (H.B == 1) coarse ? mg_setup_t<1, 2>(c, H) : mg_refresh_t<1, 2>(c, H);
    else coarse ? mg_setup_t<2, 2>(c, H) : mg_refresh_t<2, 2>(c, H);
  } else {
    if (H.B == 1) coarse ? mg_setup_t<1, 3>(c, H) : mg_refresh_t<1, 3>(c, H);
    else coarse ? mg_setup_t<3, 3>(c, H) : mg_refresh_t<3, 3>(c, H);
  }
}

// V-cycle on H's level-0 vectors (b[0] and the first sweep in x[0] set by the
// caller); the result is left in x[0].
void mg_vcycle(Ctx &c, MGHier<real> &H) {
  if (c.d == 2) {
    if (H.B == 1) vcycle_t<1, 2>(c, H, 0);
    else vcycle_t<2, 2>(c, H, 0);
  } else {
    if (H.B == 1) vcycle_t<1, 3>(c, H, 0);
    else vcycle_t<3, 3>(c, H, 0);
  }
}

}  // namespace MG_NS

// ============================================================== Schur
template <>
int schur_alloc<MG_REAL>(Ctx &c, LinSys<MG_REAL> &S) {
  using namespace MG_NS;
  const int64_t nn = c.g.nnodes;
  const int d = c.d;
  if (!S.mgA) S.mgA = new MGHier<MG_REAL>();
  if (!S.mgS) S.mgS = new MGHier<MG_REAL>();
  int rc = mg_alloc(c, *S.mgA, d);
  if (!rc) rc = mg_alloc(c, *S.mgS, 1);
  if (rc) return rc;
  if (cudaMalloc(&S.DAinv, sizeof(real) * nn * d * d) || cudaMalloc(&S.vu, sizeof(real) * nn * d) ||
      cudaMalloc(&S.B1rs, sizeof(real) * nn * d) || (c.schur_lower() && cudaMalloc(&S.vp, sizeof(real) * nn)))
    return MPM_ERR_NO_MEMORY;
  return MPM_OK;
}

template <>
void schur_free<MG_REAL>(LinSys<MG_REAL> &S) {
  using namespace MG_NS;
  if (S.mgA) { mg_free(*S.mgA); delete S.mgA; S.mgA = nullptr; }
  if (S.mgS) { mg_free(*S.mgS); delete S.mgS; S.mgS = nullptr; }
  MG_REAL *ptrs[] = {S.Aval, S.Sval, S.B1c, S.W, S.B1rs, S.DAinv, S.vu, S.B2c, S.vp};
  for (MG_REAL *p : ptrs) cudaFree(p);
  S.Aval = S.Sval = S.B1c = S.W = S.B1rs = S.DAinv = S.vu = S.B2c = S.vp = nullptr;
  if (S.gexec) cudaGraphExecDestroy(S.gexec);
  if (S.itexec) cudaGraphExecDestroy(S.itexec);
  S.gexec = S.itexec = nullptr;
  S.gkey_col = S.gkey_val = nullptr;
  S.g_x0 = S.g_zp = S.g_zu = nullptr;
  S.sub_cap = 0;
}

// Split the unscaled Jacobian (after Dirichlet elimination) into A and S and
// build both hierarchies.
template <>
int schur_setup<MG_REAL>(Ctx &c, LinSys<MG_REAL> &S, bool coarse) {
  using namespace MG_NS;
  const int64_t nn = c.g.nnodes, nnzb = c.nnzb;
  const int d = c.d;
  auto drop_graphs = [&] {  // they are captured again on next use
    if (S.gexec) cudaGraphExecDestroy(S.gexec);
    if (S.itexec) cudaGraphExecDestroy(S.itexec);
    S.gexec = S.itexec = nullptr;
  };
  if (nnzb > S.sub_cap) {
    // the captured graph reads these buffers (B1c, and Aval / Sval through
    // the finest multigrid level)
    drop_graphs();
    MG_REAL *ptrs[] = {S.Aval, S.Sval, S.B1c, S.W, S.B2c};
    for (MG_REAL *p : ptrs) cudaFree(p);
    S.Aval = S.Sval = S.B1c = S.W = S.B2c = nullptr;
    const int64_t cap = c.nnzb_cap;
    auto get = [&](MG_REAL **p, int64_t vals) { return step_malloc(c, (void **)p, sizeof(real) * vals); };
    if (get(&S.Aval, cap * d * d) || get(&S.Sval, cap) || get(&S.B1c, cap * d) || get(&S.W, cap * d) ||
        (c.schur_lower() && get(&S.B2c, cap * d))) {
      S.sub_cap = 0;
      c.last_error = "device allocation of the block preconditioner failed";
      return MPM_ERR_NO_MEMORY;
    }
    S.sub_cap = cap;
  }
  const bool full = coarse || !S.coarse_built;
  // the finest level's A P on a window of so many slots; where the new buffer does not
  // fit beside the narrower one, in its place (without either, the next set-up
  // allocates anew)
  auto reserve_ap = [&](MGHier<real> &H, int slots) -> int {
    if (H.nlev == 1 || H.ap_slots >= slots) return MPM_OK;
    const size_t bytes = sizeof(real) * H.L[0].nnodes * slots * H.B * H.B;
    real *p = nullptr;
    const bool beside = step_malloc(c, (void **)&p, bytes) == MPM_OK;
    drop_graphs();
    cudaFree(H.ap[0]);
    H.ap[0] = p;
    H.ap_slots = beside ? slots : 0;
    if (beside) return MPM_OK;
    if (const int rc = step_malloc(c, (void **)&H.ap[0], bytes)) return rc;
    H.ap_slots = slots;
    return MPM_OK;
  };
  // the window of A P from the step's largest support
  int win = 3;
  for (int k = 0; k < d; ++k) win = std::max(win, std::min(c.h_cmax[k], 4) + 1);
  for (MGHier<real> *H : {S.mgA, S.mgS}) {
    if (reserve_ap(*H, d == 2 ? (win == 5 ? 25 : 16) : (win == 5 ? 125 : 64))) {
      c.last_error = "device allocation of the block preconditioner failed";
      return MPM_ERR_NO_MEMORY;
    }
    // (coarse levels kept from an earlier set-up keep their window)
    const int cwin = !full ? H->cwin : win == 3 ? 3 : 4;
    if (H->win != win || H->cwin != cwin) {  // the captured graphs hold the other window's kernels
      drop_graphs();
      H->win = win;
      H->cwin = cwin;
    }
  }
  // B1 serves the upper order's coupling update and the DIAG_A product, B2 the
  // lower order's
  const int64_t nsl = d == 2 ? 49 : 343;
  const bool fs = c.fixed_stress();
  real *b1 = !fs || !c.schur_lower() ? S.B1c : nullptr, *b2 = c.schur_lower() ? S.B2c : nullptr;
  const double *fsd = nullptr;
  if (fs) {
    run_fs_diag(c);
    fsd = c.fsd;
  }
  auto setup_blocks = [&](auto dim) {
    constexpr int D = decltype(dim)::value;
    k_split_blocks<D><<<nblk(nnzb), TPB, 0, c.st>>>(nnzb, S.val, c.row_of, c.col, fsd, c.fixed, S.Aval, b1, b2,
                                                    S.Sval);
    UPMPM_LAUNCH(c);
    if (fs) return;
    k_diag_inv_A<D><<<nblk(nn), TPB, 0, c.st>>>(nn, c.row_ptr, c.col, S.Aval, b1, S.DAinv, S.B1rs);
    k_schur_w<D><<<nblk(nnzb), TPB, 0, c.st>>>(nnzb, c.col, S.val, S.DAinv, S.W);
    k_schur_rows<D><<<nblk(ap_threads(nn, nsl)), TPB, 0, c.st>>>(c.g.nn[0], c.g.nn[1], nn, c.row_mask, c.row_ptr,
                                                                 S.val, b1, S.W, S.Sval);
    k_schur_lump<D><<<nblk(nn), TPB, 0, c.st>>>(nn, c.row_ptr, c.col, S.val, S.W, S.B1rs, S.Sval);
    c.launches += 4;
  };
  if (d == 2) setup_blocks(std::integral_constant<int, 2>{});
  else setup_blocks(std::integral_constant<int, 3>{});
  // the coarse levels and the coarsest inverses: a new Galerkin product, or (not
  // full) the product of an earlier set-up kept, the finest levels' values,
  // block-Jacobi inverses and A P refreshed
  mg_setup(c, *S.mgA, c.row_ptr, c.col, S.Aval, 0, full);
  mg_setup(c, *S.mgS, c.row_ptr, c.col, S.Sval, d, full);
  if (full) {
    dense_invert_pair(c, *S.mgA, *S.mgS);
    S.coarse_built = true;
    S.coarse_step = c.steps;
  }
  tail_build_pair(c, *S.mgA, *S.mgS, !full);
  return check_cuda(c, cudaGetLastError(), "schur setup");
}

// z = M^{-1} v (block triangular, multigrid sub-solves) in three parts:
// split (v -> the first sub-solve's rhs and first sweep, and the other
// block's part of v), the multigrid core (first V-cycle, coupling update,
// second V-cycle), merge (-> z).  Upper order: S-cycle, B1 update, A-cycle;
// lower order: A-cycle, B2 update, S-cycle.
namespace MG_NS {
// x0: where the first sub-solve's first sweep goes (its hierarchy's x[0])
void schur_split(Ctx &c, LinSys<MG_REAL> &S, const MG_REAL *v, MG_REAL *x0) {
  const int64_t nn = c.g.nnodes;
  MGHier<real> &HS = *S.mgS, &HA = *S.mgA;
  const Geom g = geom(c, nn);
  const real *dsc = S.dscinv;  // D^-1: the unscaled v is D^-1 times the scaled one
  const real om = mg_omega(c);
  if (c.schur_lower()) {
    const real *dinv = HA.L[0].dinv;
    if (c.d == 2) launch_pdl(c, k_split_lower<2>, g.blocks, g.tpb, 0, nn, v, dsc, HA.b[0], x0, dinv, S.vp, om);
    else launch_pdl(c, k_split_lower<3>, g.blocks, g.tpb, 0, nn, v, dsc, HA.b[0], x0, dinv, S.vp, om);
    return;
  }
  const real *dinv = HS.L[0].dinv;
  if (c.d == 2) launch_pdl(c, k_split<2>, g.blocks, g.tpb, 0, nn, v, dsc, S.vu, HS.b[0], x0, dinv, om);
  else launch_pdl(c, k_split<3>, g.blocks, g.tpb, 0, nn, v, dsc, S.vu, HS.b[0], x0, dinv, om);
}

// x0 of the hierarchy whose V-cycle comes first
MG_REAL *schur_first_x0(Ctx &c, LinSys<MG_REAL> &S) { return c.schur_lower() ? S.mgA->x[0] : S.mgS->x[0]; }

void schur_core(Ctx &c, LinSys<MG_REAL> &S) {
  const int64_t nn = c.g.nnodes;
  MGHier<real> &HS = *S.mgS, &HA = *S.mgA;
  const bool large = nn >= LN_LARGE_ROWS;
  constexpr int LV = 8, LL = sizeof(real) == sizeof(double) ? 4 : 8;
  const Geom g = geom(c, nn * (large ? LL : LV));
  const int32_t *rp = c.row_ptr, *cl = c.col;
  const real om = mg_omega(c);
  if (c.schur_lower()) {
    mg_vcycle(c, HA);
    const real *b2 = S.B2c, *zu = HA.x[0], *vp = S.vp, *dinv = HS.L[0].dinv;
    auto go = [&](auto kernel) {
      launch_pdl(c, kernel, g.blocks, g.tpb, 0, nn, rp, cl, b2, zu, vp, HS.b[0], HS.x[0], dinv, om);
    };
    if (c.d == 2) large ? go(k_b2c_update<2, LL>) : go(k_b2c_update<2, LV>);
    else large ? go(k_b2c_update<3, LL>) : go(k_b2c_update<3, LV>);
    mg_vcycle(c, HS);
    return;
  }
  mg_vcycle(c, HS);
  const real *b1 = S.B1c, *zp = HS.x[0], *vu = S.vu, *dinv = HA.L[0].dinv;
  auto go = [&](auto kernel) {
    launch_pdl(c, kernel, g.blocks, g.tpb, 0, nn, rp, cl, b1, zp, vu, HA.b[0], HA.x[0], dinv, om);
  };
  if (c.d == 2) large ? go(k_b1c_update<2, LL>) : go(k_b1c_update<2, LV>);
  else large ? go(k_b1c_update<3, LL>) : go(k_b1c_update<3, LV>);
  mg_vcycle(c, HA);
}

void schur_merge(Ctx &c, LinSys<MG_REAL> &S, const MG_REAL *zu, const MG_REAL *zp, MG_REAL *z) {
  const int64_t nn = c.g.nnodes;
  const Geom g = geom(c, nn);
  if (c.d == 2) launch_pdl(c, k_merge<2>, g.blocks, g.tpb, 0, nn, zu, zp, z);
  else launch_pdl(c, k_merge<3>, g.blocks, g.tpb, 0, nn, zu, zp, z);
}
}  // namespace MG_NS

template <>
SplitP<MG_REAL> schur_split_args<MG_REAL>(Ctx &c, LinSys<MG_REAL> &S) {
  using namespace MG_NS;
  const int lower = c.schur_lower();
  MGHier<real> &H = lower ? *S.mgA : *S.mgS;
  return SplitP<MG_REAL>{S.dscinv, H.L[0].dinv, H.b[0], H.x[0], lower ? S.vp : S.vu, mg_omega(c), lower};
}

template <>
void schur_core_launch<MG_REAL>(Ctx &c, LinSys<MG_REAL> &S, const MG_REAL **zu, const MG_REAL **zp) {
  using namespace MG_NS;
  schur_core(c, S);
  *zu = S.mgA->x[0];
  *zp = S.mgS->x[0];
}

// The multigrid core is a fixed sequence of small kernels on fixed buffers: it
// is captured once into a CUDA graph and replayed between the split and merge
// kernels, which take the caller's v and z.  It is re-captured when a buffer
// it reads moves: the block columns (key below) or the Schur / multigrid
// matrices (schur_setup drops the graph when it reallocates them; a freed and
// reallocated buffer may come back at another address while col does not).
template <>
void schur_apply<MG_REAL>(Ctx &c, LinSys<MG_REAL> &S, const MG_REAL *v, MG_REAL *z) {
  using namespace MG_NS;
  if (!c.capturing && (!S.gexec || S.gkey_col != c.col || S.gkey_val != S.val ||
                       S.g_lower != (int)c.schur_lower())) {
    if (S.gexec) cudaGraphExecDestroy(S.gexec);
    S.gexec = nullptr;
    cudaGraph_t graph = nullptr;
    const int64_t before = c.launches;
    MG_REAL *x0 = schur_first_x0(c, S);
    bool ok = cudaStreamBeginCapture(c.st, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
    if (ok) {
      c.capturing = true;
      schur_core(c, S);
      c.capturing = false;
      ok = cudaStreamEndCapture(c.st, &graph) == cudaSuccess && graph;
    }
    if (ok) ok = cudaGraphInstantiate(&S.gexec, graph, 0) == cudaSuccess;
    if (graph) cudaGraphDestroy(graph);
    S.gkernels = c.launches - before;
    c.launches = before;
    if (ok) {
      S.g_x0 = x0;
      S.g_lower = (int)c.schur_lower();
      S.g_zp = S.mgS->x[0];
      S.g_zu = S.mgA->x[0];
      S.gkey_col = c.col;
      S.gkey_val = S.val;
    } else {  // capture unavailable: launch directly from now on
      cudaGetLastError();
      S.gexec = nullptr;
    }
  }
  if (S.gexec && !c.capturing) {
    schur_split(c, S, v, S.g_x0);
    cudaGraphLaunch(S.gexec, c.st);
    c.launches += S.gkernels;
    schur_merge(c, S, S.g_zu, S.g_zp, z);
    return;
  }
  schur_split(c, S, v, schur_first_x0(c, S));
  schur_core(c, S);
  schur_merge(c, S, S.mgA->x[0], S.mgS->x[0], z);
}
