// sm_103a kernels of the interior point method: residuals, diagonal update, right-hand side,
// the matrix-free PCG iteration, direction recovery, ratio test and update.
//
// Operator (the condensed form of the paper's KKT matvec, Section 4.1.1 / Listing 1):
//     K p = R^T (omega o (R p)) + Hs p + (h0 + sigma) o p,
// where R = [F; A_csr] and omega = w_R + theta placed on the constraint rows, so that
// R^T diag(omega) R = F^T W F + A^T Theta A.  One PCG iteration is two streaming passes:
// k_op_rows (row gather over R) and k_op_cols (row gather over the stored transpose R^T).
// Sums over the grid are block parts added in block order, by the last block to arrive or by every
// block of the kernel that needs them; maxima and minima, where the order does not matter, are
// taken on the integer pipe.  Results are bitwise reproducible for a fixed problem size.
#include <algorithm>
#include <cmath>

#include "state.h"

namespace ipmk {

static __device__ __forceinline__ int gwarp() { return (blockIdx.x * blockDim.x + threadIdx.x) >> 5; }
static __device__ __forceinline__ int nwarps() { return (gridDim.x * blockDim.x) >> 5; }

// Lanes per row of the streaming row kernels (see group_row_dot): G is a template parameter,
// picked per matrix at ipm_set_qp (Dev::g_rows for R, Dev::g_cols for R^T).
template <int G>
static __device__ __forceinline__ int glane() { return threadIdx.x & (G - 1); }

// Grid-stride loop over rows, G lanes per row, with a warp-uniform trip count (the group
// shuffles need every lane of the warp): the loop runs over the first row of each warp's
// groups; a group whose row is past the end works on an empty row.
#define FOR_GROUP_ROWS(G, r, ok, nrows)                                                                \
  for (int64_t r##_0 = (int64_t)gwarp() * (32 / G); r##_0 < (nrows); r##_0 += (int64_t)nwarps() * (32 / G)) \
    for (int64_t r = r##_0 + (threadIdx.x & 31) / G, r##_once = 0; r##_once == 0; r##_once = 1)           \
      for (bool ok = r < (nrows), ok##_once = true; ok##_once; ok##_once = false)

// Instantiates a launch for the lane-group size g (4, 8, 16 or 32) chosen at run time.
#define DISPATCH_G(g, ...)                         \
  do {                                             \
    switch (g) {                                   \
      case 4: { constexpr int G = 4; __VA_ARGS__; } break;   \
      case 8: { constexpr int G = 8; __VA_ARGS__; } break;   \
      case 16: { constexpr int G = 16; __VA_ARGS__; } break; \
      default: { constexpr int G = 32; __VA_ARGS__; } break; \
    }                                              \
  } while (0)


Geo make_geo(const Dev& d) {
  // at most 8 blocks of 256 threads per SM (the row kernels are grid-stride loops)
  const int cap = std::min(kMaxRedBlocks, 8 * (d.sm_count > 0 ? d.sm_count : 148));
  auto blocks_for = [cap](int64_t items, int per_block) -> int {
    int64_t b = (items + per_block - 1) / per_block;
    if (b > cap) b = cap;
    return (int)b;
  };
  Geo g;
  const int gr = d.g_rows > 0 ? d.g_rows : 32, gc = d.g_cols > 0 ? d.g_cols : 32;
  g.gR = blocks_for(d.nR, kBlock / gr);
  g.gM = blocks_for(d.m, kBlock / gr);
  g.gN = blocks_for(d.n, kBlock / gc);
  g.eM = blocks_for(d.m, kBlock);
  g.eN = blocks_for(d.n, kBlock);
  // the PCG column kernels are limited to 40 registers (6 blocks per SM): one full wave
  g.gNc = (int)std::min<int64_t>(g.gN, 6 * (int64_t)(d.sm_count > 0 ? d.sm_count : 148));
  g.gRc = (int)std::min<int64_t>(g.gR, 6 * (int64_t)(d.sm_count > 0 ? d.sm_count : 148));
  g.gR64 = (int)std::min<int64_t>(g.gR, kOpRowsMinBlocks * (int64_t)(d.sm_count > 0 ? d.sm_count : 148));
  g.gN64 = (int)std::min<int64_t>(g.gN, kOpColsMinBlocks * (int64_t)(d.sm_count > 0 ? d.sm_count : 148));
  // the residual and right-hand-side column kernels are limited to 64 registers (4 per SM)
  g.gNr = (int)std::min<int64_t>(g.gN, 4 * (int64_t)(d.sm_count > 0 ? d.sm_count : 148));
  return g;
}

// ------------------------------------------------------------------------------ low-rank term

// H's low-rank term U W U^T (eq:bfgs_hessian: H = H0 + U W U^T, U dense n x 2k, W diagonal) is
// applied matrix-free in two dense passes over U: t = U^T v (this pair of kernels, a
// reduction over the n rows of U split into row chunks, one partial vector per block, summed
// in block order), then (U (W t))_j inside the column kernels (lr_row).  Row-major U makes
// both passes read rows of U contiguously.
//
// A thread owns 8 columns (in 16-byte loads of two where rows start on 16 bytes; neighbouring
// threads load neighbouring ones) and walks every rg-th row of its block's chunk, rg = 256 /
// ceil(ucols / 8) rows of threads side by side: of 256 threads 250 carry columns at 200 columns,
// where 32 lanes over 128-column slices carried 200 of 256 values, and every float64 instruction of
// a warp costs the same.  (n = 77373, 200 columns: 41 us before.)  The rg partial sums of a column are added by as
// many threads as there are for it: by one thread a column they were a serial chain of 256 at up to
// 8 columns (both kernels at n = 20000, 7 columns: 20.9 -> 15.0 us; n = 1000, one column: 20.9 -> 10.8).
constexpr int kLrCols = 8;
constexpr int kLrTile = kBlock / 4;              // rows of U a block of the column pass takes at a time
constexpr int kLrSlice = 256 * kLrCols;          // columns a block covers at a time
template <bool VEC>
__global__ void __launch_bounds__(256) k_lr_part(Dev d, const double* __restrict__ v) {
  __shared__ double sh[256][kLrCols + 1];
  const int64_t uc = d.ucols, n = d.n;
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  const int64_t j0 = (int64_t)blockIdx.x * per, j1 = j0 + per < n ? j0 + per : n;
  const int tid = threadIdx.x;
  for (int64_t r0 = 0; r0 < uc; r0 += kLrSlice) {
    const int w = (int)(uc - r0 < kLrSlice ? uc - r0 : kLrSlice);
    const int nch = (w + kLrCols - 1) / kLrCols, rg = 256 / nch;
    const int c = tid % nch, g = tid / nch;
    const int nv = w / 2;                  // VEC: pairs of columns
    double acc[kLrCols];
#pragma unroll
    for (int k = 0; k < kLrCols; ++k) acc[k] = 0.0;
    if (g < rg) {
      if (VEC) {
        const double2* u = reinterpret_cast<const double2*>(d.U + r0) + c;
        const int64_t uv = uc / 2;
        int64_t j = j0 + g;
        if (c + (kLrCols / 2 - 1) * nch < nv) {
          for (; j + rg < j1; j += 2 * rg) {
            const double2 *p0 = u + j * uv, *p1 = u + (j + rg) * uv;
            double2 a[kLrCols / 2], b[kLrCols / 2];
            const double x0 = __ldg(v + j), x1 = __ldg(v + j + rg);
#pragma unroll
            for (int k = 0; k < kLrCols / 2; ++k) a[k] = __ldg(p0 + k * nch);
#pragma unroll
            for (int k = 0; k < kLrCols / 2; ++k) b[k] = __ldg(p1 + k * nch);
#pragma unroll
            for (int k = 0; k < kLrCols / 2; ++k) {
              acc[2 * k] = fma(a[k].x, x0, acc[2 * k]);
              acc[2 * k + 1] = fma(a[k].y, x0, acc[2 * k + 1]);
            }
#pragma unroll
            for (int k = 0; k < kLrCols / 2; ++k) {
              acc[2 * k] = fma(b[k].x, x1, acc[2 * k]);
              acc[2 * k + 1] = fma(b[k].y, x1, acc[2 * k + 1]);
            }
          }
        }
        for (; j < j1; j += rg) {
          const double x0 = __ldg(v + j);
#pragma unroll
          for (int k = 0; k < kLrCols / 2; ++k)
            if (c + k * nch < nv) {
              const double2 a = __ldg(u + j * uv + k * nch);
              acc[2 * k] = fma(a.x, x0, acc[2 * k]);
              acc[2 * k + 1] = fma(a.y, x0, acc[2 * k + 1]);
            }
        }
      } else {
        const double* u = d.U + r0 + c;
        for (int64_t j = j0 + g; j < j1; j += rg) {
          const double x0 = __ldg(v + j);
#pragma unroll
          for (int k = 0; k < kLrCols; ++k)
            if (c + k * nch < w) acc[k] = fma(__ldg(u + j * uc + k * nch), x0, acc[k]);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kLrCols; ++k) sh[tid][k] = acc[k];
    __syncthreads();
    // column t by L neighbouring threads (L w <= 256), then a tree over them
    const int L = nch > 16 ? 1 : 1 << (31 - __clz(32 / nch));
    for (int t = tid / L; t - (tid & 31) / L < w; t += 256 / L) {   // whole warps: the shuffles need them
      // the thread and accumulator of column t
      const int i = VEC ? t / 2 : t, th = i % nch, k = VEC ? 2 * (i / nch) + (t & 1) : i / nch;
      double s = 0.0;
      if (t < w)
        for (int q = tid & (L - 1); q < rg; q += L) s += sh[q * nch + th][k];
      for (int o = L / 2; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (t < w && (tid & (L - 1)) == 0)
        d.upart[(r0 + t) * (int64_t)d.ublocks + blockIdx.x] = s;   // column-major: the final sum reads runs
    }
    __syncthreads();
  }
}

// lrs = uw o t, t_r = the sum of the block partials of column r (stored column-major; a block of
// four warps per column: thread l adds the partials of blocks l, l + 128, ..., then a fixed tree);
// quad: lrq_r = uw_r t_r^2.  (608 parts a column: 4.4 us with a warp a column, 3.2 us.)
constexpr int kLrFinal = 128;
__global__ void __launch_bounds__(kLrFinal) k_lr_final(Dev d, int quad) {
  __shared__ double sh[32];
  for (int64_t r = blockIdx.x; r < d.ucols; r += gridDim.x) {
    double t = 0.0;
    for (int b = threadIdx.x; b < d.ublocks; b += kLrFinal) t += d.upart[r * (int64_t)d.ublocks + b];
    t = block_sum0(t, sh);
    if (threadIdx.x == 0) {
      const double sv = d.uw[r] * t;
      d.lrs[r] = sv;
      if (quad) d.lrq[r] = sv * t;
    }
    __syncthreads();
  }
}

cudaError_t launch_lr(const Dev& d, const double* v, int quad, cudaStream_t st) {
  if (!d.ucols) return cudaSuccess;
  if (d.ucols & 1) k_lr_part<false><<<d.ublocks, 256, 0, st>>>(d, v);
  else k_lr_part<true><<<d.ublocks, 256, 0, st>>>(d, v);
  k_lr_final<<<(int)std::min<int64_t>(d.ucols, 4096), kLrFinal, 0, st>>>(d, quad);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ setup

// diag(H)_j = h0_j + sum_i w_R,i R_ij^2 + sum_r uw_r U_jr^2 + Hs_jj  (computed once; Section
// 4.1.2 caches it).
__global__ void k_diagH(Dev d) {
  for (int64_t j = gwarp(); j < d.n; j += nwarps()) {
    double acc = warp_row_dot<true>(d.RT_ptr[j], d.RT_ptr[j + 1], d.RT_idx, d.RT_val, d.wR);
    if (d.ucols) {
      double ul = 0.0;
      for (int64_t r = threadIdx.x & 31; r < d.ucols; r += 32) {
        const double u = d.U[j * d.ucols + r];
        ul = fma(d.uw[r] * u, u, ul);
      }
      acc += warp_sum(ul);
    }
    double hjj = 0.0;
    if (d.Hs_ptr) {
      for (int64_t e = d.Hs_ptr[j] + (threadIdx.x & 31); e < d.Hs_ptr[j + 1]; e += 32)
        if (d.Hs_idx[e] == j) hjj += d.Hs_val[e];
      hjj = warp_sum(hjj);
    }
    if ((threadIdx.x & 31) == 0) d.diagH[j] = d.h0[j] + acc + hjj;
  }
}

// repeats = 1 where a constraint row repeats a column (rows increase within a column of A^T, so the
// entries lie side by side).
__global__ void k_find_repeats(Dev d) {
  for (int64_t j = gwarp(); j < d.n; j += nwarps())
    for (int64_t e = d.AT_ptr[j] + 1 + (threadIdx.x & 31); e < d.AT_ptr[j + 1]; e += 32)
      if (d.AT_idx[e] == d.AT_idx[e - 1]) d.sc->repeats = 1;
}

cudaError_t launch_find_repeats(const Dev& d, cudaStream_t st) {
  if (!d.m || !d.nnzA) return cudaSuccess;
  k_find_repeats<<<(int)std::min<int64_t>((d.n + 7) / 8, 4096), kBlock, 0, st>>>(d);
  return cudaGetLastError();
}

__global__ void k_fill_rowk(Dev d) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < d.nR; r += (int64_t)gridDim.x * blockDim.x)
    d.rowk[r] = -1;
}

__global__ void k_fill_rowk2(Dev d) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x)
    d.rowk[d.arow[k]] = (int32_t)k;
}

// rowk: the constraint index of each row of R (-1 for rows of the factor alone).
cudaError_t launch_fill_rowk(const Dev& d, cudaStream_t st) {
  if (!d.nR) return cudaSuccess;
  const int b = (int)std::min<int64_t>((d.nR + kBlock - 1) / kBlock, 4096);
  k_fill_rowk<<<b, kBlock, 0, st>>>(d);
  if (d.m) k_fill_rowk2<<<(int)std::min<int64_t>((d.m + kBlock - 1) / kBlock, 4096), kBlock, 0, st>>>(d);
  return cudaGetLastError();
}

cudaError_t launch_diagH(const Dev& d, cudaStream_t st) {
  Geo g = make_geo(d);
  if (g.gN) k_diagH<<<g.gN, kBlock, 0, st>>>(d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ residuals

// t = R x; v = w_R o t; y placed on the constraint rows of R (0 on the others); partial sum of
// w_R t^2 (the factor part of x^T H x).  Rows in the order of k_op_rows and as many blocks resident
// (n = 50000: 145 -> 130 us).
template <int G>
__global__ void __launch_bounds__(256, kOpRowsMinBlocks) k_rows_resid(Dev d, double* part) {
  __shared__ double sh[32];
  double acc = 0.0;
  FOR_GROUP_ROWS(G, ri, ok, d.nR) {
    const int64_t r = (ok && d.rperm) ? (int64_t)d.rperm[ri] : ri;   // as in k_op_rows
    const int64_t beg = ok ? d.R_ptr[r] : 0, end = ok ? d.R_ptr[r + 1] : 0;
    const double t = group_row_dot<G, false>(beg, end, glane<G>(), d.R_idx, d.R_val, d.x);
    if (ok && glane<G>() == 0) {
      const double w = d.wR[r];
      const int32_t k = d.rowk[r];
      d.tR[r] = t;
      d.vR[r] = w * t;
      d.vR2[r] = k >= 0 ? d.y[k] : 0.0;
      acc = fma(w * t, t, acc);
    }
  }
  acc = block_sum0(acc, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = acc;
}

// A running maximum of numbers >= 0 kept as the bits of the float64 (their order is the
// numbers'), so that its reductions run on the integer pipe; negative numbers and NaN are
// passed over, as fmax does.
__device__ __forceinline__ void keep_max(long long& m, double v) {
  const long long b = __double_as_longlong(v);
  if (b > m && b <= 0x7ff0000000000000ll) m = b;
}
__device__ __forceinline__ void keep_abs_max(long long& m, double v) { keep_max(m, fabs(v)); }
__device__ __forceinline__ long long warp_imax(long long m) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long t = __shfl_xor_sync(0xffffffffu, m, o);
    m = t > m ? t : m;
  }
  return m;
}

// Slots of the partials of a residual summary: rows (RS_XFX), constraint rows, variables.
enum ResidSlot { RS_XFX = 0, RS_RP = 1, RS_VIOL = 2, RS_RS = 3, RS_BY = 4, RS_SY = 5, RS_RD = 6, RS_HX = 7,
                 RS_ATY = 8, RS_RC = 9, RS_XHX = 10, RS_CX = 11, RS_LU = 12, RS_TZ = 14, RS_BVIOL = 15,
                 RS_YMAX = 28, RS_CERT = 29, RS_ZMAX = 30 };

// Constraint rows (block b of nb): r_p = A x + s - b, r_s = s o y - mu and their scalar parts.
__device__ void cons_resid(const Dev& d, double* part, int b, int nb) {
  __shared__ long long sm[4][8];
  __shared__ double sh[2][8];
  const double mu = d.sc->mu;
  long long rp_inf = 0, viol = 0, rs_inf = 0, ymax = 0;
  double by = 0.0, sy = 0.0;
  for (int64_t k = b * (int64_t)kBlock + threadIdx.x; k < d.m; k += (int64_t)nb * kBlock) {
    const double ax = d.tR[d.arow[k]], s = d.s[k], y = d.y[k], bk = d.b[k];
    const double rp = ax + s - bk;
    d.rp[k] = rp;
    keep_abs_max(rp_inf, rp);
    keep_max(viol, ax - bk);
    keep_abs_max(rs_inf, s * y - mu);
    by = fma(bk, y, by);
    keep_abs_max(ymax, y);
    sy = fma(s, y, sy);
  }
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  rp_inf = warp_imax(rp_inf);
  viol = warp_imax(viol);
  rs_inf = warp_imax(rs_inf);
  ymax = warp_imax(ymax);
  by = warp_sum(by);
  sy = warp_sum(sy);
  if (lane == 0) {
    sm[0][w] = rp_inf; sm[1][w] = viol; sm[2][w] = rs_inf; sm[3][w] = ymax;
    sh[0][w] = by; sh[1][w] = sy;
  }
  __syncthreads();
  if (w == 0) {
    const int q = lane >> 3, i = lane & 7;
    long long m = sm[q][i];
    double v = q < 2 ? sh[q][i] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const long long t = __shfl_xor_sync(0xffffffffu, m, o);
      m = t > m ? t : m;
      v += __shfl_xor_sync(0xffffffffu, v, o);
    }
    const int mslot[4] = {RS_RP, RS_VIOL, RS_RS, RS_YMAX}, sslot[2] = {RS_BY, RS_SY};
    if (i == 0) {
      part[mslot[q] * kMaxRedBlocks + b] = __longlong_as_double(m);
      if (q < 2) part[sslot[q] * kMaxRedBlocks + b] = v;
    }
  }
}

// Variables: Hx = R^T vR + Hs x + h0 o x, A^T y (over the stored A^T, y placed on R rows in
// vR2), r_d and the scalar parts of the objective, the dual objective and the complementarity
// sum; the blocks from gcols on take the constraint rows.
//
// A float64 instruction holds a quarter of an SM for 64 cycles whatever its lanes do, so the
// per-variable arithmetic (some 20 instructions) is not done by one lane in G: the groups leave
// their sums in shared memory and the block's 256 / G variables are finished by that many
// neighbouring threads.  The two dot products share one tree (each half of a group carries one
// of them after the first exchange).  The maxima are reduced as integers.  n = 7001 at 16 lanes:
// 31 us as one kernel of one-lane epilogues and twelve float64 block reductions (and 7 us for
// the constraint rows), 9.8 us for both so.
template <int G>
__global__ void __launch_bounds__(256, 4) k_cols_resid(Dev d, double* part, int gcols) {
  if ((int)blockIdx.x >= gcols) {
    cons_resid(d, part, (int)blockIdx.x - gcols, (int)gridDim.x - gcols);
    return;
  }
  constexpr int C = kBlock / G;        // variables a block handles per trip
  constexpr int S = 32 / G;            // of them per warp
  __shared__ double st[2][4][C];
  __shared__ double sw[4][8];
  __shared__ long long sm[7][2];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gl = glane<G>(), c = tid / G;
  const double mu = d.sc->mu;
  long long rd_inf = 0, hx_inf = 0, aty_inf = 0, rc_inf = 0, bviol = 0, cert = 0, zmax = 0;
  double xHsx = 0.0, cx = 0.0, lu = 0.0, tz = 0.0;
  int buf = 0;
  for (int64_t j0 = (int64_t)blockIdx.x * C; j0 < d.n; j0 += (int64_t)gcols * C, buf ^= 1) {
    const int64_t j = j0 + c;
    const bool ok = j < d.n;
    double a = group_row_part<G>(ok ? d.RT_ptr[j] : 0, ok ? d.RT_ptr[j + 1] : 0, gl, d.RT_idx, d.RT_val, d.vR);
    double b = group_row_part<G>(ok ? d.AT_ptr[j] : 0, ok ? d.AT_ptr[j + 1] : 0, gl, d.AT_idx, d.AT_val, d.vR2);
    // lower half of the group: the sum of a, upper half: of b
    const bool up = gl & (G / 2);
    const double keep = up ? b : a, give = up ? a : b;
    double t = keep + __shfl_xor_sync(0xffffffffu, give, G / 2);
#pragma unroll
    for (int o = G / 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (gl == 0) st[buf][0][c] = t;
    if (gl == G / 2) st[buf][1][c] = t;
    if (d.Hs_ptr) {
      const double hs = group_row_dot<G, false>(ok ? d.Hs_ptr[j] : 0, ok ? d.Hs_ptr[j + 1] : 0, gl, d.Hs_idx, d.Hs_val, d.x);
      if (gl == 0) st[buf][2][c] = hs;
    }
    if (d.ucols) {
      const double lr = lr_row<G>(d, j, ok, gl);
      if (gl == 0) st[buf][3][c] = lr;
    }
    __syncthreads();
    const int64_t jj = j0 + tid;
    if (tid < C && jj < d.n) {
      const double xj = d.x[jj], zl = d.zl[jj], zu = d.zu[jj], cj = d.c[jj];
      const double hsx = (d.Hs_ptr ? st[buf][2][tid] : 0.0) + d.h0[jj] * xj;
      const double hx = st[buf][0][tid] + hsx + (d.ucols ? st[buf][3][tid] : 0.0);
      const double aty = st[buf][1][tid];
      const double rd = hx + cj + aty - zl + zu;
      d.rd[jj] = rd;
      keep_abs_max(cert, aty - zl + zu);
      keep_abs_max(zmax, zl);
      keep_abs_max(zmax, zu);
      keep_abs_max(rd_inf, rd);
      keep_abs_max(hx_inf, hx);
      keep_abs_max(aty_inf, aty);
      xHsx = fma(xj, hsx, xHsx);
      cx = fma(cj, xj, cx);
      if (d.fl[jj]) {
        const double l = d.l[jj], tl = xj - l;
        keep_abs_max(rc_inf, tl * zl - mu);
        lu = fma(l, zl, lu);
        tz = fma(tl, zl, tz);
        keep_max(bviol, -tl);
      }
      if (d.fu[jj]) {
        const double u = d.u[jj], tu = u - xj;
        keep_abs_max(rc_inf, tu * zu - mu);
        lu = fma(-u, zu, lu);
        tz = fma(tu, zu, tz);
        keep_max(bviol, -tu);
      }
    }
  }
  // sums over the block in the order of a 256-thread block whose groups' first lanes hold the
  // values: over the S groups of a warp, then over the 8 warps
  constexpr int NW = (C + 31) / 32;    // warps that hold values
  if (w < NW) {
    double v[4] = {xHsx, cx, lu, tz};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int o = S / 2; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
      if (tid < C && (tid & (S - 1)) == 0) sw[q][tid / S] = v[q];
    }
    long long m[7] = {rd_inf, hx_inf, aty_inf, rc_inf, bviol, cert, zmax};
#pragma unroll
    for (int q = 0; q < 7; ++q) {
      m[q] = warp_imax(m[q]);
      if (lane == 0) sm[q][w] = m[q];
    }
  }
  __syncthreads();
  if (w == 0) {
    double v = sw[lane >> 3][lane & 7];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    const int sslot[4] = {RS_XHX, RS_CX, RS_LU, RS_TZ};
    if ((lane & 7) == 0) part[sslot[lane >> 3] * kMaxRedBlocks + blockIdx.x] = v;
    const int mslot[7] = {RS_RD, RS_HX, RS_ATY, RS_RC, RS_BVIOL, RS_CERT, RS_ZMAX};
    if (lane < 7) {
      const long long m = NW > 1 && sm[lane][1] > sm[lane][0] ? sm[lane][1] : sm[lane][0];
      part[mslot[lane] * kMaxRedBlocks + blockIdx.x] = __longlong_as_double(m);
    }
  }
}

static __device__ void set_eta(Scal* sc);
static __device__ void control_step(const Dev& d, double cg_rel, cudaGraphConditionalHandle h, int set_cond);

// One block: totals of the partials, one warp per quantity, then the relative KKT residual
// (primal, dual, gap), the objective values and the norm of the mu test.
//   primal = max(viol_A, viol_bounds) / (1 + ||b||), dual = ||r_d|| / (1 + max(||c||, ||Hx||, ||A^T y||)),
//   gap = |pobj - dobj| / (1 + |pobj| + |dobj|),
//   ||r||_mu = max(||r_s, r_l, r_u||, (1 + |pobj|) / N_c * max(||r_p|| / (1 + ||b||), ||r_d|| / (1 + ||c||))).
// All its quotients are formed by one division, a lane each.
// MODE RSM_START: also the complementarity mean (the start points' mu); RSM_CONTROL: also the
// iteration's control step.  (24.6 us with every thread over all 19 quantities in turn and one
// thread's chain of nine divisions, plus 4.4 us and a launch for the control; 5 us so, 8 to 12 us
// with the control step.)
constexpr int kFinalThreads = 640;
template <int MODE>
__global__ void __launch_bounds__(kFinalThreads) k_resid_final(Dev d, int gR, int gM, int gN, const double* part,
                                                              cudaGraphConditionalHandle h, int set_cond) {
  constexpr int NM = 11, NS = 5;
  __shared__ double mx[NM], sum[NS + 1], comp[2][16];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int mslot[NM] = {RS_RP, RS_VIOL, RS_RS, RS_YMAX, RS_RD, RS_HX, RS_ATY, RS_RC, RS_BVIOL, RS_CERT, RS_ZMAX};
  const int sslot[NS] = {RS_XFX, RS_BY, RS_XHX, RS_CX, RS_LU};
  if (w < NS) {                                   // sums: warps 0..4
    const int nb = w == 0 ? gR : (w == 1 ? gM : gN);
    const double* p = part + sslot[w] * kMaxRedBlocks;
    double acc = 0.0;
    for (int b = lane; b < nb; b += 128) {
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = b + 32 * k < nb ? p[b + 32 * k] : 0.0;
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (b - lane + 32 * k < nb) acc += v[k];
    }
    acc = warp_sum(acc);
    if (lane == 0) sum[w] = acc;
  } else if (w < NS + NM) {                       // maxima: warps 5..15
    const int q = w - NS, nb = q < 4 ? gM : gN;
    const double* p = part + mslot[q] * kMaxRedBlocks;
    long long m = 0;
    for (int b = lane; b < nb; b += 32) keep_max(m, p[b]);
    m = warp_imax(m);
    if (lane == 0) mx[q] = __longlong_as_double(m);
  } else if (w == NS + NM && d.ucols) {           // x^T U W U^T x
    double q = 0.0;
    for (int64_t r = lane; r < d.ucols; r += 32) q += d.lrq[r];
    q = warp_sum(q);
    if (lane == 0) sum[NS] = q;
  }
  if (MODE == RSM_START) {
    // the complementarity sums, added as 512 threads over the blocks, by warps, then warp by warp
    __syncthreads();
    if (w < 16) {
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int nb = q == 0 ? gM : gN;
        const double* p = part + (q == 0 ? RS_SY : RS_TZ) * kMaxRedBlocks;
        double v = 0.0;
        for (int b = threadIdx.x; b < nb; b += 512) v += p[b];
        v = warp_sum(v);
        if (lane == 0) comp[q][w] = v;
      }
    }
  }
  __syncthreads();
  if (w > 0) return;
  Scal* sc = d.sc;
  const double xHx = sum[0] + sum[2] + (d.ucols ? sum[NS] : 0.0);
  const double pobj = 0.5 * xHx + sum[3];
  const double by = sum[1], dobj = -0.5 * xHx - by + sum[4];
  const double bn = sc->bnorm, cn = sc->cnorm;
  const double nc = sc->ncomp > 0 ? (double)sc->ncomp : 1.0;
  const double mi = fmax(d.m ? mx[3] : 0.0, mx[10]);
  double num = 0.0, den = 1.0;
  switch (lane) {
    case 0: num = fmax(mx[1], mx[8]); den = 1.0 + bn; break;                       // primal
    case 1: num = mx[4]; den = 1.0 + fmax(cn, fmax(mx[5], mx[6])); break;          // dual
    case 2: num = fabs(pobj - dobj); den = 1.0 + fabs(pobj) + fabs(dobj); break;   // gap
    case 3: num = mx[0]; den = 1.0 + bn; break;
    case 4: num = mx[4]; den = 1.0 + cn; break;
    case 5: num = mx[9]; den = mi > 0.0 ? mi : 1.0; break;
    case 6: num = by - sum[4]; den = mi > 0.0 ? mi : 1.0; break;
    case 7: num = 1.0 + fabs(pobj); den = nc; break;
    case 8:
      if (MODE == RSM_CONTROL) {
        num = sc->rr;
        den = sc->rhs2 > 0.0 ? sc->rhs2 : 1.0;
      }
      break;
    case 9:
      if (MODE == RSM_START) {
        double sy = 0.0, tz = 0.0;
        for (int i = 0; i < 16; ++i) {
          sy += comp[0][i];
          tz += comp[1][i];
        }
        num = sy + tz;
        den = nc;
      }
      break;
    default: break;
  }
  const double quot = num / den;
  double cg_rel = 0.0;
  if (MODE == RSM_CONTROL) cg_rel = sqrt(__shfl_sync(0xffffffffu, quot, 8));
  const double primal = __shfl_sync(0xffffffffu, quot, 0), dual = __shfl_sync(0xffffffffu, quot, 1),
               gap = __shfl_sync(0xffffffffu, quot, 2), ep = __shfl_sync(0xffffffffu, quot, 3),
               ed = __shfl_sync(0xffffffffu, quot, 4), cres = __shfl_sync(0xffffffffu, quot, 5),
               cgap = __shfl_sync(0xffffffffu, quot, 6), sf = __shfl_sync(0xffffffffu, quot, 7),
               cmean = __shfl_sync(0xffffffffu, quot, 9);
  if (lane == 0) {
    sc->res_primal = primal;
    sc->res_dual = dual;
    sc->res_gap = gap;
    double rk = fmax(primal, fmax(dual, gap));
    if (!isfinite(rk)) rk = INFINITY;
    sc->rel_kkt = rk;
    sc->pobj = pobj;
    sc->dobj = dobj;
    sc->rp_inf = mx[0];
    sc->rd_inf = mx[4];
    const double rc = fmax(mx[2], mx[7]);
    sc->rc_inf = rc;
    sc->rnorm_mu = fmax(rc, sf * fmax(ep, ed));
    if (MODE == RSM_START) sc->comp_mean = cmean;
    sc->mult_inf = mi;
    sc->cert_res = mi > 0.0 ? cres : INFINITY;
    sc->cert_gap = mi > 0.0 ? cgap : 0.0;
    if (MODE == RSM_CONTROL) control_step(d, sc->rhs2 > 0.0 ? cg_rel : 0.0, h, set_cond);
    if (MODE == RSM_STEP) {
      set_eta(sc);
      if (sc->eta_asked > 0.0) sc->eta = sc->eta_asked;
    }
  }
}

cudaError_t launch_residual_summary(const Dev& d, const Geo& g, cudaStream_t st, int mode, cudaGraphConditionalHandle h) {
  double* part = d.partials;
  if (d.nR) DISPATCH_G(d.g_rows, k_rows_resid<G><<<g.gR64, kBlock, 0, st>>>(d, part));
  launch_lr(d, d.x, 1, st);
  const int gM = d.m ? g.eM : 0;
  DISPATCH_G(d.g_cols, k_cols_resid<G><<<g.gNr + gM, kBlock, 0, st>>>(d, part, g.gNr));
  const int gR = d.nR ? g.gR64 : 0, sc = h != 0 ? 1 : 0;
  if (mode == RSM_START) k_resid_final<RSM_START><<<1, kFinalThreads, 0, st>>>(d, gR, gM, g.gNr, part, h, sc);
  else if (mode == RSM_CONTROL) k_resid_final<RSM_CONTROL><<<1, kFinalThreads, 0, st>>>(d, gR, gM, g.gNr, part, h, sc);
  else if (mode == RSM_STEP) k_resid_final<RSM_STEP><<<1, kFinalThreads, 0, st>>>(d, gR, gM, g.gNr, part, h, sc);
  else k_resid_final<RSM_PLAIN><<<1, kFinalThreads, 0, st>>>(d, gR, gM, g.gNr, part, h, sc);
  return cudaGetLastError();
}

// Complementarity residuals as vectors (for the step-level query): r_s into ds, r_l into dzl,
// r_u into dzu.
__global__ void k_comp_resid(Dev d) {
  const double mu = d.sc->mu;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x)
    d.ds[k] = d.s[k] * d.y[k] - mu;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * blockDim.x) {
    d.dzl[j] = d.fl[j] ? (d.x[j] - d.l[j]) * d.zl[j] - mu : 0.0;
    d.dzu[j] = d.fu[j] ? (d.u[j] - d.x[j]) * d.zu[j] - mu : 0.0;
  }
}

cudaError_t launch_comp_resid(const Dev& d, const Geo& g, cudaStream_t st) {
  k_comp_resid<<<std::max(g.eN, g.eM), kBlock, 0, st>>>(d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ start point

// x0 = 0 projected into the box shrunk by delta_j = 0.1 min(1, (u_j - l_j) / 2) (0.1 for a
// one-sided bound; 0 for a free variable).
__global__ void k_start_x(Dev d) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * blockDim.x) {
    const bool fl = d.fl[j], fu = d.fu[j];
    const double width = (fl && fu) ? d.u[j] - d.l[j] : 2.0;
    const double delta = 0.1 * fmin(1.0, 0.5 * width);
    double x = 0.0;
    if (fl) x = fmax(x, d.l[j] + delta);
    if (fu) x = fmin(x, d.u[j] - delta);
    d.x[j] = x;
  }
}

// s0 = max(b - A x0, 1)   (tR holds R x0)
__global__ void k_start_s(Dev d) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x)
    d.s[k] = fmax(d.b[k] - d.tR[d.arow[k]], 1.0);
}

// g = H x0 + c; z_l0 = max(1, g), z_u0 = max(1, -g) on finite bounds.
template <int G>
__global__ void k_start_z(Dev d) {
  FOR_GROUP_ROWS(G, j, ok, d.n) {
    const int64_t beg = ok ? d.RT_ptr[j] : 0, end = ok ? d.RT_ptr[j + 1] : 0;
    const double hx = group_row_dot<G, false>(beg, end, glane<G>(), d.RT_idx, d.RT_val, d.vR);
    double hs = 0.0;
    if (d.Hs_ptr) {
      const int64_t hb = ok ? d.Hs_ptr[j] : 0, he = ok ? d.Hs_ptr[j + 1] : 0;
      hs = group_row_dot<G, false>(hb, he, glane<G>(), d.Hs_idx, d.Hs_val, d.x);
    }
    if (d.ucols) hs += lr_row<G>(d, j, ok, glane<G>());
    if (ok && glane<G>() == 0) {
      const double g = hx + hs + d.h0[j] * d.x[j] + d.c[j];
      d.zl[j] = d.fl[j] ? fmax(1.0, g) : 0.0;
      d.zu[j] = d.fu[j] ? fmax(1.0, -g) : 0.0;
    }
  }
}

// y0 = 1 on every row (theta starts moderate: no constraint row begins stiff).
__global__ void k_start_y(Dev d) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x)
    d.y[k] = 1.0;
}

__global__ void k_start_mu(Dev d) {
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    Scal* sc = d.sc;
    sc->mu0 = sc->comp_mean > 0.0 ? sc->comp_mean : 1.0;
    sc->mu0_cold = sc->mu0;
    sc->mu = sc->mu0;
    sc->ipm_iter = 0;
    sc->stop = 0;
    sc->status = DS_RUNNING;
    set_eta(sc);
  }
}

cudaError_t launch_start_point(const Dev& d, const Geo& g, cudaStream_t st) {
  k_start_x<<<g.eN, kBlock, 0, st>>>(d);
  if (d.nR) DISPATCH_G(d.g_rows, k_rows_resid<G><<<g.gR64, kBlock, 0, st>>>(d, d.partials));
  if (d.m) k_start_s<<<g.eM, kBlock, 0, st>>>(d);
  launch_lr(d, d.x, 0, st);
  DISPATCH_G(d.g_cols, k_start_z<G><<<g.gN, kBlock, 0, st>>>(d));
  if (d.m) k_start_y<<<g.eM, kBlock, 0, st>>>(d);
  cudaError_t e = launch_residual_summary(d, g, st, RSM_START);
  if (e != cudaSuccess) return e;
  k_start_mu<<<1, 32, 0, st>>>(d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ control

// Inexact-Newton forcing term of the PCG solve: ||r|| <= eta ||rhs|| with
// eta = clamp(eta_factor * relKKT, eta_min, eta_max) (reading; the paper states no tolerance).
static __device__ void set_eta(Scal* sc) {
  double e = sc->eta_factor * sc->rel_kkt;
  if (!(e <= sc->eta_max)) e = sc->eta_max;
  if (e < sc->eta_min) e = sc->eta_min;
  sc->eta = e;
}

// Algorithm 1's tail on the device: stop when rel KKT <= tol (reading of "mu <= mu_tol"),
// else mu <- mu / 10 when ||r|| < mu; then the PCG tolerance eta for the next Newton step.  One
// thread, at the end of the residual summary; cg_rel: ||r|| / ||rhs|| of the step's PCG.
static __device__ void control_step(const Dev& d, double cg_rel, cudaGraphConditionalHandle h, int set_cond) {
  Scal* sc = d.sc;
  sc->ipm_iter += 1;
  const double rk = sc->rel_kkt;
  const double mu_step = sc->mu;
  const int refine = d.storage != ST_F64 ? sc->refine_it : 0;
  sc->cg_total += sc->cg_iter;
  sc->refine_total += refine;
  if (sc->cg_iter > sc->max_cg_step) sc->max_cg_step = sc->cg_iter;
  // PCG stall: the PCG of two consecutive Newton steps ended at the iteration limit with a
  // residual above 1e-2 of its right-hand side (worse than the loosest tolerance the method
  // asks for).  A direction that misses a tight tolerance but is otherwise accurate is kept
  // (inexact Newton): the paper's doubly augmented system under Jacobi PCG lives there.
  sc->cg_fail_run = (sc->cg_conv || cg_rel <= 1e-2) ? 0 : sc->cg_fail_run + 1;
  if (sc->status == DS_RUNNING && sc->cg_fail_run >= 2) sc->status = DS_CG_STALL;
  if (sc->status == DS_NUMERICAL || sc->status == DS_CG_STALL || sc->status == DS_TIMEOUT) {
    sc->stop = 1;
  } else if (sc->ipm_iter >= 5 && !(sc->res_primal <= sc->tol_kkt) && sc->mult_inf > 1e10 &&
             isfinite(sc->mult_inf) && sc->cert_res <= 1e-8 && sc->cert_gap < -1e-8) {
    // the multipliers diverge along a Farkas certificate of primal infeasibility:
    // y >= 0, z >= 0 with A^T y - z_l + z_u ~ 0 and b^T y - l^T z_l + u^T z_u < 0
    sc->stop = 1;
    sc->status = DS_INFEASIBLE;
  } else if (!isfinite(rk) || !isfinite(sc->pobj)) {
    sc->stop = 1;
    sc->status = DS_NUMERICAL;
  } else if (rk <= sc->tol_kkt) {
    sc->stop = 1;
    sc->status = DS_OK;
  } else if (sc->ipm_iter >= sc->max_ipm) {
    sc->stop = 1;
    sc->status = DS_MAX_ITER;
  } else if (sc->rnorm_mu < sc->mu) {
    sc->mu = fmax(sc->mu * 0.1, sc->mu0 * 1e-16);
  }
  set_eta(sc);
  if (d.trace && sc->trace_rows < sc->trace_cap) {
    double* t = d.trace + (int64_t)sc->trace_rows * kTraceCols;
    t[0] = sc->ipm_iter; t[1] = mu_step; t[2] = rk; t[3] = sc->res_primal; t[4] = sc->res_dual;
    t[5] = sc->res_gap; t[6] = sc->alpha_p; t[7] = sc->alpha_d; t[8] = sc->cg_iter; t[9] = sc->cg_conv;
    t[10] = sc->n_stiff; t[11] = cg_rel; t[12] = sc->eta_used; t[13] = refine;
    sc->trace_rows += 1;
  }
  if (set_cond) cudaGraphSetConditional(h, sc->stop ? 0u : 1u);
}

__global__ void k_ask_eta(Dev d, double eta) {
  if (threadIdx.x == 0) d.sc->eta_asked = eta;
}

cudaError_t launch_ask_eta(const Dev& d, double eta, cudaStream_t st) {
  k_ask_eta<<<1, 32, 0, st>>>(d, eta);
  return cudaGetLastError();
}

// Start of a solve on the device: per-solve totals and the trace cleared.
__global__ void k_solve_begin(Dev d) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  Scal* sc = d.sc;
  sc->cg_total = 0;
  sc->refine_total = 0;
  sc->max_cg_step = 0;
  sc->trace_rows = 0;
  sc->max_stiff_seen = 0;
  sc->fallback_total = 0;
  sc->cg_fail_run = 0;
  sc->stop = 0;
  sc->status = DS_RUNNING;
}

cudaError_t launch_solve_begin(const Dev& d, cudaStream_t st) {
  k_solve_begin<<<1, 32, 0, st>>>(d);
  return cudaGetLastError();
}

// Warm start from the current iterate: mu0 = its complementarity mean (after a residual summary).
__global__ void k_warm_mu(Dev d) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  Scal* sc = d.sc;
  sc->mu0 = sc->comp_mean > 0.0 ? sc->comp_mean : 1.0;
  sc->mu = sc->mu0;
  sc->ipm_iter = 0;
  set_eta(sc);
}

// Warm start (reading; the paper warm-starts the SQP's QPs, Section 3.2, without a recipe):
// every complementarity pair of the previous solution is raised to at least
// mu_w = warm_rho * mu0_cold (mu0 of the last cold start on this handle): s and y scaled
// together by sqrt(mu_w / (s y)), z_l, z_u raised to mu_w / t.  No shift before a cold start.
__global__ void k_warm_shift(Dev d) {
  const double muw = d.sc->warm_rho * d.sc->mu0_cold;
  if (!(muw > 0.0)) return;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x) {
    const double sy = d.s[k] * d.y[k];
    if (sy < muw) {
      const double f = sqrt(muw / fmax(sy, 1e-300));
      d.s[k] *= f;
      d.y[k] *= f;
    }
  }
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * blockDim.x) {
    if (d.fl[j]) d.zl[j] = fmax(d.zl[j], muw / (d.x[j] - d.l[j]));
    if (d.fu[j]) d.zu[j] = fmax(d.zu[j], muw / (d.u[j] - d.x[j]));
  }
}

cudaError_t launch_warm_start(const Dev& d, const Geo& g, cudaStream_t st) {
  k_warm_shift<<<std::max(g.eN, g.eM), kBlock, 0, st>>>(d);
  cudaError_t e = launch_residual_summary(d, g, st, RSM_START);
  if (e != cudaSuccess) return e;
  k_warm_mu<<<1, 32, 0, st>>>(d);
  return cudaGetLastError();
}

__global__ void k_set_cond(cudaGraphConditionalHandle h, unsigned v) {
  if (threadIdx.x == 0 && blockIdx.x == 0) cudaGraphSetConditional(h, v);
}

cudaError_t launch_set_cond(cudaGraphConditionalHandle h, unsigned v, cudaStream_t st) {
  k_set_cond<<<1, 32, 0, st>>>(h, v);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ diagonal update

// The diagonals of the Newton step and what its right-hand side has on the rows of R, in one
// launch (six before: two copies, a fill and three kernels, 2-4 us each at n = 7001):
//   theta = y / s; omega = w_R + theta and thR = theta on the constraint rows (w_R and 0 on the
//   others; twice theta for the doubly augmented system, whose (1,1) block carries
//   2 B^T D^-1 B = 2 A^T Theta A); u = theta o r_p - r_s / s placed on the rows (vR2);
//   sigma = z_l / t_l + z_u / t_u; M0 = diag(H) + sigma; Minv = 1 / M0 until the Jacobi diagonal
//   of the moderate rows replaces it.
// Constraint rows are walked by constraint, not by row of R: a quotient costs a warp the same
// for one lane as for 32, and the constraint rows lie scattered among R's.  Also clears the
// step lengths' minima and the variables' stiff-row masks.
__global__ void k_diag(Dev d) {
  const double mu = d.sc->mu;
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, dt = (int64_t)gridDim.x * blockDim.x;
  if (t0 < 2) d.sc->step_min[t0] = kInfBits;
  for (int64_t i = t0; i < d.n * d.sc_words; i += dt) d.sc_mask[i] = 0u;
  for (int64_t r = t0; r < d.nR; r += dt)
    if (d.rowk[r] < 0) {
      d.omega[r] = d.wR[r];
      d.thR[r] = 0.0;
      d.vR2[r] = 0.0;
    }
  for (int64_t k = t0; k < d.m; k += dt) {
    const double s = d.s[k], y = d.y[k], rp = d.rp[k];
    const double th = y / s;
    const int32_t row = d.arow[k];
    d.theta[k] = th;
    const double thf = d.aug ? 2.0 * th : th;
    d.omega[row] = d.wR[row] + thf;
    d.thR[row] = thf;
    const double rs = s * y - mu;
    const double u = th * rp - rs / s;                // theta o r2, r2 = r_p - r_s / y
    d.vR2[row] = d.aug ? 2.0 * u : u;
    if (d.aug) {
      // eq:2x2_augmented: top r1 + 2 B^T D^-1 r2 = r1 - 2 A^T (theta o r2); bottom r2;
      // Jacobi on the bottom block D = s / y: 1 / D = theta
      const double r2 = rp - rs / y;
      d.rhs[d.n + k] = r2;
      d.r[d.n + k] = r2;
      d.dx[d.n + k] = 0.0;
      d.Minv[d.n + k] = th;
    }
  }
  for (int64_t j = t0; j < d.n; j += dt) {
    double sg = 0.0;
    if (d.fl[j]) sg += d.zl[j] / (d.x[j] - d.l[j]);
    if (d.fu[j]) sg += d.zu[j] / (d.u[j] - d.x[j]);
    d.sigma[j] = sg;
    const double m0 = d.diagH[j] + sg;
    d.M0[j] = m0;
    d.Minv[j] = 1.0 / m0;
  }
}

cudaError_t launch_diag_update(const Dev& d, const Geo& g, cudaStream_t st) {
  const int64_t most = std::max(d.n, std::max(d.nR / 4, d.m));   // the rows' part is a fill
  const int cap = 8 * (d.sm_count > 0 ? d.sm_count : 148);
  k_diag<<<(int)std::max<int64_t>(1, std::min<int64_t>((most + kBlock - 1) / kBlock, cap)), kBlock, 0, st>>>(d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ Jacobi

// M_j = M0_j + sum_k A_kj^2 thR_k  (thR: theta of the constraint rows kept in the diagonal part;
// the factor rows' part w_R is already in M0 through diag(H)).
// Writes 1 / M_j to out (INV) or M_j.
template <bool INV, int G>
__global__ void k_jacobi(Dev d, double* out) {
  FOR_GROUP_ROWS(G, j, ok, d.n) {
    const int64_t beg = ok ? d.AT_ptr[j] : 0, end = ok ? d.AT_ptr[j + 1] : 0;
    const double a = group_row_dot<G, true>(beg, end, glane<G>(), d.AT_idx, d.AT_val, d.thR);
    if (ok && glane<G>() == 0) {
      const double mj = d.M0[j] + a;
      out[j] = INV ? 1.0 / mj : mj;
    }
  }
}

cudaError_t launch_jacobi_full(const Dev& d, const Geo& g, double* out, cudaStream_t st) {
  DISPATCH_G(d.g_at, k_jacobi<false, G><<<g.gN, kBlock, 0, st>>>(d, out));
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ stiff rows

// Half-octave bin of y = ratio / gamma > 1, floor(2 log2 y), from the float64's exponent and
// whether its mantissa reaches sqrt 2 (float64 log2 takes some forty instructions a warp).
__device__ __forceinline__ int half_octave(double y) {
  const long long b = __double_as_longlong(y);
  const int e = (int)(b >> 52) - 1023;
  const int bin = 2 * e + ((b & 0xfffffffffffffll) >= 0x6a09e667f3bcdll ? 1 : 0);
  return bin < 0 ? 0 : (bin >= kHistBins ? kHistBins - 1 : bin);
}

// The stiff rows, in one launch: ratio_k = theta_k sum_j A_kj^2 / M0_j of every constraint row,
// a histogram of the ratios above gamma in half-octave bins and the list of those rows; the last
// block picks the smallest threshold bin whose count from the top stays <= stiff_max, takes the
// listed rows at or above it, orders them by constraint and gives each its slot (thR = 0: its
// theta leaves the Jacobi part).  Only listed rows are looked at again: a pass of one block
// over all m took 8 us at m = 3500 and 133 us at m = 68618.
template <int G>
__global__ void k_stiff_select(Dev d) {
  __shared__ unsigned int h[kHistBins];
  __shared__ int list[1024];                       // stiff_max's limit
  __shared__ int s_cnt;
  __shared__ double s_thr;
  __shared__ bool s_last;
  Scal* sc = d.sc;
  for (int i = threadIdx.x; i < kHistBins; i += blockDim.x) h[i] = 0u;
  __syncthreads();
  const double gamma = sc->stiff_gamma;
  FOR_GROUP_ROWS(G, k, ok, d.m) {
    const int32_t row = ok ? d.arow[k] : 0;
    const int64_t beg = ok ? d.R_ptr[row] : 0, end = ok ? d.R_ptr[row + 1] : 0;
    // sum_j R_kj^2 / M0_j with 1 / M0 precomputed in Minv
    const double acc = group_row_dot<G, true>(beg, end, glane<G>(), d.R_idx, d.R_val, d.Minv);
    if (ok && glane<G>() == 0) {
      const double ratio = d.theta[k] * acc;
      if (ratio > gamma) {
        d.ratio[k] = ratio;
        d.cand[atomicAdd(&sc->n_cand, 1)] = (int32_t)k;
        atomicAdd(&h[half_octave(ratio / gamma)], 1u);
      }
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < kHistBins; i += blockDim.x)
    if (h[i]) atomicAdd(&d.hist[i], h[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&sc->ticket[T_HIST], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < 32) {
    // lane l: bins 63 - 2l and 62 - 2l; counts from the top by a scan over the lanes
    const unsigned c1 = __ldcg(&d.hist[63 - 2 * lane]), c0 = __ldcg(&d.hist[62 - 2 * lane]);
    unsigned cum = c1 + c0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned t = __shfl_up_sync(0xffffffffu, cum, o);
      if (lane >= o) cum += t;
    }
    const unsigned cap = (unsigned)sc->stiff_max;
    int cut = kHistBins;                           // no stiff rows
    if (cum - c0 <= cap) cut = 63 - 2 * lane;
    if (cum <= cap) cut = 62 - 2 * lane;
    cut = __reduce_min_sync(0xffffffffu, cut);
    if (lane == 0) {
      // rows in bins >= cut are stiff: threshold = gamma * 2^(cut/2)
      s_thr = cut >= kHistBins ? INFINITY : (cut == 0 ? gamma : gamma * exp2(0.5 * cut));
      s_cnt = 0;
    }
  }
  __syncthreads();
  const double thr = s_thr;
  const int nc = *(volatile int*)&sc->n_cand;
  for (int i = tid; i < nc; i += blockDim.x) {
    const int32_t k = __ldcg(&d.cand[i]);
    if (__ldcg(&d.ratio[k]) >= thr) {
      const int at = atomicAdd(&s_cnt, 1);
      if (at < 1024) list[at] = k;
    }
  }
  __syncthreads();
  const int total = min(s_cnt, 1024), ns = min(total, d.stiff_cap);
  for (int i = tid; i < total; i += blockDim.x) {
    const int k = list[i];
    int rank = 0;
    for (int q = 0; q < total; ++q) rank += list[q] < k ? 1 : 0;
    if (rank < ns) {
      const int32_t row = d.arow[k];
      d.stiff_k[rank] = k;
      d.st_beg[rank] = d.R_ptr[row];
      d.st_end[rank] = d.R_ptr[row + 1];
      d.thR[row] = 0.0;
    }
  }
  for (int i = tid; i < kHistBins; i += blockDim.x) d.hist[i] = 0u;
  if (tid == 0) {
    sc->stiff_thresh = thr;
    sc->n_stiff = ns;
    sc->sc_used = 0;
    if (ns > sc->max_stiff_seen) sc->max_stiff_seen = ns;
    sc->n_cand = 0;
    sc->ticket[T_HIST] = 0u;
  }
}

// Stiff entries per variable, built from the stiff rows alone (a pass over A^T for the counts, a
// one-block scan and a second pass took 21 us at n = 7001 and 53 us at n = 50000): each entry
// (slot a, variable j) sets bit a of j's mask; the masks' counts give every variable a run of
// the list; an entry's place in its run is the number of lower bits, so a run holds its slots in
// increasing order.  (Runs are handed out in any order; nothing depends on where a run lies.)  A column
// that a row repeats has one place, with the entries' sum, as the operator has it (Dev::repeats).
__global__ void k_sc_mask(Dev d) {
  const int ns = d.sc->n_stiff, lane = threadIdx.x & 31;
  for (int a = gwarp(); a < ns; a += nwarps())
    for (int64_t e = d.st_beg[a] + lane; e < d.st_end[a]; e += 32)
      atomicOr(&d.sc_mask[(int64_t)d.R_idx[e] * d.sc_words + (a >> 5)], 1u << (a & 31));
}

__global__ void k_sc_runs(Dev d) {
  if (d.sc->n_stiff == 0) return;
  const int lane = threadIdx.x & 31;
  for (int64_t j0 = (int64_t)blockIdx.x * blockDim.x; j0 < d.n; j0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = j0 + threadIdx.x;
    int cnt = 0;
    if (j < d.n)
      for (int w = 0; w < d.sc_words; ++w) cnt += __popc(d.sc_mask[j * d.sc_words + w]);
    int cum = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, cum, o);
      if (lane >= o) cum += t;
    }
    int base = 0;
    if (lane == 31 && cum) base = atomicAdd(&d.sc->sc_used, cum);
    base = __shfl_sync(0xffffffffu, base, 31) + cum - cnt;
    if (j < d.n) {
      const int run = base + cnt <= d.sc_cap ? cnt : 0;
      d.sc_run[j] = make_int2(base, run);
      if (d.repeats)
        for (int t = 0; t < run; ++t) d.sc_val[base + t] = 0.0;
    }
  }
}

__global__ void k_sc_fill(Dev d) {
  const int ns = d.sc->n_stiff, lane = threadIdx.x & 31;
  for (int a = gwarp(); a < ns; a += nwarps())
    for (int64_t e = d.st_beg[a] + lane; e < d.st_end[a]; e += 32) {
      const int64_t j = d.R_idx[e];
      const unsigned* m = d.sc_mask + j * d.sc_words;
      const int2 run = d.sc_run[j];
      int at = __popc(m[a >> 5] & ((1u << (a & 31)) - 1u));
      for (int w = 0; w < (a >> 5); ++w) at += __popc(m[w]);
      if (at < run.y) {
        d.sc_slot[run.x + at] = a;
        if (d.repeats) atomicAdd(&d.sc_val[run.x + at], d.R_val[e]);
        else d.sc_val[run.x + at] = d.R_val[e];
      }
    }
}

// G = Theta_s^{-1} + A_s M^{-1} A_s^T (dense, n_stiff x n_stiff, leading dimension stiff_cap).
// One block per stiff row a, one thread per slot b: for every entry (j, R_aj) of the row in
// order, thread b adds (R_aj / M_j) A_bj if bit b of j's mask is set.  The row's entries, masks
// and the variables' runs are staged in shared memory 256 entries at a time, so what remains is
// each slot's chain of additions.  (With a barrier per entry: 27 us at n = 7001, 42 entries a
// row; 87 us at n = 50000, 250 a row.)
constexpr int kGramEntries = 256, kGramItems = 2048, kGramSlots = 4;   // 4 * 256 slots = stiff_max's limit
__global__ void __launch_bounds__(256) k_gram_G(Dev d) {
  extern __shared__ unsigned gm[];               // masks [word][entry], then ranks before a word [word][entry]
  __shared__ double f[kGramEntries], lv[kGramItems];
  __shared__ int base[kGramEntries], off[kGramEntries + 1], wsum[8];
  const int ns = d.sc->n_stiff, a = blockIdx.x;
  if (a >= ns) return;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int words = (ns + 31) >> 5;
  unsigned short* pre = reinterpret_cast<unsigned short*>(gm + (size_t)words * kGramEntries);
  double acc[kGramSlots] = {0.0, 0.0, 0.0, 0.0};
  const int64_t beg = d.st_beg[a], end = d.st_end[a];
  for (int64_t e0 = beg; e0 < end; e0 += kGramEntries) {
    const int ne = (int)(end - e0 < kGramEntries ? end - e0 : kGramEntries);
    int cnt = 0;
    if (tid < ne) {
      const int64_t j = d.R_idx[e0 + tid];
      f[tid] = d.R_val[e0 + tid] * d.Minv[j];
      const int2 run = d.sc_run[j];
      base[tid] = run.x;
      cnt = run.y;
      int p = 0;
      for (int q = 0; q < words; ++q) {
        const unsigned m = cnt ? d.sc_mask[j * d.sc_words + q] : 0u;
        gm[q * kGramEntries + tid] = m;
        pre[q * kGramEntries + tid] = (unsigned short)p;
        p += __popc(m);
      }
    }
    int cum = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, cum, o);
      if (lane >= o) cum += t;
    }
    if (lane == 31) wsum[w] = cum;
    __syncthreads();
    int before = 0;
    for (int q = 0; q < w; ++q) before += wsum[q];
    off[tid] = before + cum - cnt;
    if (tid == 255) off[256] = before + cum;
    __syncthreads();
    const int items = off[kGramEntries];
    const bool staged = items <= kGramItems;
    if (staged)
      for (int i = tid; i < items; i += 256) {
        int lo = 0, hi = kGramEntries;             // the last entry whose run starts at or before i
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (off[mid] <= i) lo = mid;
          else hi = mid;
        }
        lv[i] = d.sc_val[base[lo] + i - off[lo]];
      }
    __syncthreads();
#pragma unroll
    for (int g = 0; g < kGramSlots; ++g) {
      const int q = w + 8 * g;                     // the mask word of this warp's slots
      if (q < words)
        for (int e = 0; e < ne; ++e) {
          const unsigned m = gm[q * kGramEntries + e];
          if (m >> lane & 1u) {
            const int at = pre[q * kGramEntries + e] + __popc(m & ((1u << lane) - 1u));
            acc[g] = fma(f[e], staged ? lv[off[e] + at] : d.sc_val[base[e] + at], acc[g]);
          }
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int g = 0; g < kGramSlots; ++g) {
    const int b = tid + 256 * g;
    if (b < ns) d.G[(int64_t)a * d.stiff_cap + b] = b == a ? acc[g] + 1.0 / d.theta[d.stiff_k[a]] : acc[g];
  }
}

// ------------------------------------------------------------------------------ rhs

// PCG start from ||rhs||^2: tolerance eta^2 ||rhs||^2, counters reset.
static __device__ void finish_rhs(Scal* sc, double rhs2) {
  sc->rhs2 = rhs2;
  sc->eta_used = sc->eta;
  sc->tol2 = sc->eta * sc->eta * rhs2;
  sc->cg_iter = 0;
  sc->cg_conv = 0;
  sc->cg_done = (rhs2 == 0.0 || !isfinite(rhs2)) ? 1 : 0;
  if (!isfinite(rhs2)) sc->status = DS_NUMERICAL;
  else if (rhs2 == 0.0) sc->cg_conv = 1;
}

// A lane's parts of sum_k A_kj u_k (plain) and sum_k A_kj^2 thR_k (squared): the right-hand side
// and the Jacobi diagonal read the same entries of A^T.
template <int G, bool SQ>
__device__ __forceinline__ void group_plain_sq_part(const int64_t beg, const int64_t end, const int gl,
                                                    const int32_t* __restrict__ idx, const double* __restrict__ val,
                                                    const double* __restrict__ xp, const double* __restrict__ xs,
                                                    double& op, double& os) {
  double a = 0.0, b = 0.0, a1 = 0.0, b1 = 0.0;
  int64_t e = beg + gl;
  for (; e + G < end; e += 2 * G) {
    const double v0 = __ldg(val + e), v1 = __ldg(val + e + G);
    const int i0 = __ldg(idx + e), i1 = __ldg(idx + e + G);
    a = fma(v0, __ldg(xp + i0), a);
    if (SQ) b = fma(v0 * v0, __ldg(xs + i0), b);
    a1 = fma(v1, __ldg(xp + i1), a1);
    if (SQ) b1 = fma(v1 * v1, __ldg(xs + i1), b1);
  }
  if (e < end) {
    const double v0 = __ldg(val + e);
    const int i0 = __ldg(idx + e);
    a = fma(v0, __ldg(xp + i0), a);
    if (SQ) b = fma(v0 * v0, __ldg(xs + i0), b);
  }
  op = a + a1;
  os = b + b1;
}

// rhs = -r_d - r_l / t_l + r_u / t_u - A^T u (u = vR2 on the constraint rows) and, with JAC, the
// Jacobi diagonal's inverse; PCG start r = rhs, dx = 0; ||rhs||^2.  As in k_cols_resid the groups
// leave their sums in shared memory and the block's 256 / G variables are finished by as many
// neighbouring threads (four quotients each: one lane in G doing them cost 12 of 63 us at n =
// 50000), and the two sums share one tree.
template <int G, bool JAC>
__global__ void __launch_bounds__(256, 4) k_rhs(Dev d) {
  constexpr int C = kBlock / G;
  constexpr int NW = (C + 31) / 32;
  __shared__ double st[2][2][C];
  __shared__ double sh[32];
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, gl = glane<G>(), c = tid / G;
  const double mu = d.sc->mu;
  double r2 = 0.0;
  int buf = 0;
  for (int64_t j0 = (int64_t)blockIdx.x * C; j0 < d.n; j0 += (int64_t)gridDim.x * C, buf ^= 1) {
    const int64_t j = j0 + c;
    const bool ok = j < d.n;
    double a, b;
    group_plain_sq_part<G, JAC>(ok ? d.AT_ptr[j] : 0, ok ? d.AT_ptr[j + 1] : 0, gl, d.AT_idx, d.AT_val, d.vR2, d.thR, a, b);
    if (JAC) {
      const bool up = gl & (G / 2);
      const double keep = up ? b : a, give = up ? a : b;
      a = keep + __shfl_xor_sync(0xffffffffu, give, G / 2);
    } else {
      a += __shfl_xor_sync(0xffffffffu, a, G / 2);
    }
#pragma unroll
    for (int o = G / 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (gl == 0) st[buf][0][c] = a;
    if (JAC && gl == G / 2) st[buf][1][c] = a;
    __syncthreads();
    const int64_t jj = j0 + tid;
    if (tid < C && jj < d.n) {
      if (JAC) d.Minv[jj] = 1.0 / (d.M0[jj] + st[buf][1][tid]);
      double g = -d.rd[jj] - st[buf][0][tid];
      const double xj = d.x[jj];
      if (d.fl[jj]) { const double tl = xj - d.l[jj]; g -= (tl * d.zl[jj] - mu) / tl; }
      if (d.fu[jj]) { const double tu = d.u[jj] - xj; g += (tu * d.zu[jj] - mu) / tu; }
      d.rhs[jj] = g;
      d.r[jj] = g;
      d.dx[jj] = 0.0;
      r2 = fma(g, g, r2);
    }
  }
  if (JAC && d.aug)   // the bottom block's right-hand side (written by k_diag)
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x)
      r2 = fma(d.rhs[d.n + k], d.rhs[d.n + k], r2);
  // ||rhs||^2: block parts, added by the last block
  if ((JAC && d.aug) || w < NW) r2 = warp_sum(r2);
  if (lane == 0) sh[w] = r2;
  __syncthreads();
  double* part = d.partials + 20 * kMaxRedBlocks;
  if (tid == 0) {
    const int nw = JAC && d.aug ? kBlock / 32 : NW;
    double t = sh[0];
    for (int i = 1; i < nw; ++i) t += sh[i];
    part[blockIdx.x] = t;
    __threadfence();
    s_last = atomicAdd(&d.sc->ticket[T_INIT], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last || w > 0) return;
  __threadfence();
  double t = 0.0;
  for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + b);
  t = warp_sum(t);
  if (lane == 0) {
    d.sc->ticket[T_INIT] = 0u;
    finish_rhs(d.sc, t);
  }
}

cudaError_t launch_rhs(const Dev& d, const Geo& g, int precond, cudaStream_t st) {
  // one block per 256 / g_at variables, at most the four per SM the kernel is compiled for
  const int gat = d.g_at > 0 ? d.g_at : 32;
  const int64_t want = (d.n * gat + kBlock - 1) / kBlock;
  const int nb = (int)std::min<int64_t>(want, 4 * (int64_t)(d.sm_count > 0 ? d.sm_count : 148));
  if (precond == PC_DENSE) {
    DISPATCH_G(d.g_at, k_rhs<G, false><<<nb, kBlock, 0, st>>>(d));
  } else {
    DISPATCH_G(d.g_at, k_rhs<G, true><<<nb, kBlock, 0, st>>>(d));
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ PCG

// v = omega o (R p).  MODE 0: inside PCG (skips once converged); MODE 1: single apply;
// MODE 2: single apply when the reduced-precision PCG asks for a residual replacement.
template <int MODE, int G>
__global__ void __launch_bounds__(256, kOpRowsMinBlocks) k_op_rows(Dev d) {
  if (MODE == 0 && d.sc->cg_done) return;
  if (MODE == 2 && !d.sc->ru_do) return;
  FOR_GROUP_ROWS(G, ri, ok, d.nR) {
    // rows in windows ordered by length (rperm), so the groups of one warp run equal trips
    const int64_t r = (ok && d.rperm) ? (int64_t)d.rperm[ri] : ri;
    const int64_t beg = ok ? d.R_ptr[r] : 0, end = ok ? d.R_ptr[r + 1] : 0;
    const double t = group_row_dot_u<G, 2>(beg, end, glane<G>(), d.R_idx, d.R_val, d.p);
    if (ok && glane<G>() == 0) {
      double v = d.omega[r] * t;
      if (MODE == 0 && d.aug) {
        // doubly augmented: top gets -A^T p_bottom; bottom q = B p_top + D p_bottom
        const int32_t k = d.rowk[r];
        if (k >= 0) {
          const double pb = d.p[d.n + k];
          v -= pb;
          d.q[d.n + k] = -t + pb * (d.s[k] / d.y[k]);
        }
      }
      d.vR[r] = v;
    }
  }
}

// v = omega o (R p) over the pieces of R's rows (FP64; one descriptor per piece of a run
// instead of one index per entry); otherwise as k_op_rows.
template <int MODE, int G>
__global__ void __launch_bounds__(256, 6) k_op_rows_runs(Dev d) {
  if (MODE == 0 && d.sc->cg_done) return;
  FOR_GROUP_ROWS(G, ri, ok, d.nR) {
    const int64_t r = (ok && d.rperm) ? (int64_t)d.rperm[ri] : ri;
    double a = 0.0;
    for_row_pieces<G>(d, r, ok, glane<G>(), [&](int64_t e, int c) { a = fma(__ldg(d.R_val + e), __ldg(d.p + c), a); });
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    const double t = a;
    if (ok && glane<G>() == 0) {
      double v = d.omega[r] * t;
      if (MODE == 0 && d.aug) {
        const int32_t k = d.rowk[r];
        if (k >= 0) {
          const double pb = d.p[d.n + k];
          v -= pb;
          d.q[d.n + k] = -t + pb * (d.s[k] / d.y[k]);
        }
      }
      d.vR[r] = v;
    }
  }
}

cudaError_t launch_op_rows_runs(const Dev& d, const Geo& g, int mode, cudaStream_t st) {
  if (!d.nR) return cudaSuccess;
  if (mode == 0) DISPATCH_G(d.g_rows, k_op_rows_runs<0, G><<<g.gRc, kBlock, 0, st>>>(d));
  else DISPATCH_G(d.g_rows, k_op_rows_runs<1, G><<<g.gRc, kBlock, 0, st>>>(d));
  return cudaGetLastError();
}

// q = R^T v + Hs p + (h0 + sigma) o p; p^T q by blocks.
// MODE 0: inside PCG; MODE 1: a single operator apply (no scalars touched); MODE 2: as 1,
// when the reduced-precision PCG asks for a residual replacement.
// EXT: with any of a sparse block of H, the low-rank term and the augmented system; without, the
// pass keeps its registers for the loads (six blocks an SM allow 40; no form spills).
// The block's 256 / G variables are finished by that many neighbouring threads: the last
// float64 instructions of a variable cost a warp the same for one lane as for 32 (n = 50000,
// 49.9 million entries: 132 -> 119 us with both; the entries' multiply-adds alone take 84 us of
// the float64 pipe).
template <int MODE, int G, bool EXT>
__global__ void __launch_bounds__(256, kOpColsMinBlocks) k_op_cols(Dev d) {
  constexpr int C = kBlock / G;
  __shared__ double sh[32];
  __shared__ double st[2][C];
  if (MODE == 0 && d.sc->cg_done) return;
  if (MODE == 2 && !d.sc->ru_do) return;
  const int tid = threadIdx.x, gl = glane<G>();
  double pq = 0.0;
  int buf = 0;
  for (int64_t j0 = (int64_t)blockIdx.x * C; j0 < d.n; j0 += (int64_t)gridDim.x * C, buf ^= 1) {
    const int64_t j = j0 + tid / G;
    const bool ok = j < d.n;
    const int64_t beg = ok ? d.RT_ptr[j] : 0, end = ok ? d.RT_ptr[j + 1] : 0;
    double acc = group_row_dot<G, false>(beg, end, gl, d.RT_idx, d.RT_val, d.vR);
    if (EXT && d.Hs_ptr) {
      const int64_t hb = ok ? d.Hs_ptr[j] : 0, he = ok ? d.Hs_ptr[j + 1] : 0;
      acc += group_row_dot<G, false>(hb, he, gl, d.Hs_idx, d.Hs_val, d.p);
    }
    if (EXT && d.ucols) acc += lr_row<G, true>(d, j, ok, gl);
    if (gl == 0) st[buf][tid / G] = acc;
    __syncthreads();
    const int64_t jj = j0 + tid;
    if (tid < C && jj < d.n) {
      const double pj = d.p[jj];
      const double qj = st[buf][tid] + (d.h0[jj] + d.sigma[jj]) * pj;
      d.q[jj] = qj;
      pq = fma(pj, qj, pq);
    }
  }
  if (MODE != 0) return;
  if (EXT && d.aug)   // p^T q over the bottom block too (q's bottom written by the rows pass)
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x)
      pq = fma(d.p[d.n + k], d.q[d.n + k], pq);
  store_pq_part(d, pq, sh);
}

// The same where H has the low-rank term alone (no matrix rows, no sparse block; float64 storage,
// an even number of columns): a block takes kLrTile rows of U at a time, four lanes a row, four
// 16-byte loads of U in flight a lane, and finishes its rows by that many neighbouring threads.
// n = 77373, 200 columns: 45.9 us in the general kernel, 38.2 here; the float64 pipe alone takes
// 26 us, U (124 MB, the size of the L2) 18 us from memory.  Loading the next four pairs ahead of
// the adds at 64 registers a thread was slower (42.8 us).
template <int MODE>
__global__ void __launch_bounds__(256, kOpColsMinBlocks) k_op_cols_lr(Dev d) {
  constexpr int G = 4, B = 4;
  __shared__ double sh[32];
  __shared__ double st[2][kLrTile];
  if (MODE == 0 && d.sc->cg_done) return;
  const int tid = threadIdx.x, gl = tid & (G - 1), c = tid / G;
  const int nv = (int)(d.ucols >> 1);
  const double2* s2 = reinterpret_cast<const double2*>(d.lrs);
  double pq = 0.0;
  int buf = 0;
  for (int64_t j0 = (int64_t)blockIdx.x * kLrTile; j0 < d.n; j0 += (int64_t)gridDim.x * kLrTile, buf ^= 1) {
    const int64_t j = j0 + c < d.n ? j0 + c : d.n - 1;
    const double2* row = reinterpret_cast<const double2*>(d.U + j * d.ucols);
    double a0 = 0.0, a1 = 0.0;
    for (int v = gl; v < nv; v += B * G) {
      double2 u[B], w[B];
#pragma unroll
      for (int k = 0; k < B; ++k) {
        const bool in = v + k * G < nv;
        u[k] = in ? __ldg(row + v + k * G) : make_double2(0.0, 0.0);
        w[k] = in ? __ldg(s2 + v + k * G) : make_double2(0.0, 0.0);
      }
#pragma unroll
      for (int k = 0; k < B; ++k)
        if (v - gl + k * G < nv) {     // the same for the whole group: no float64 work past the row's end
          a0 = fma(u[k].x, w[k].x, a0);
          a1 = fma(u[k].y, w[k].y, a1);
        }
    }
    a0 += a1;
    a0 += __shfl_xor_sync(0xffffffffu, a0, 2);
    a0 += __shfl_xor_sync(0xffffffffu, a0, 1);
    if (gl == 0) st[buf][c] = a0;
    __syncthreads();
    const int64_t jj = j0 + tid;
    if (tid < kLrTile && jj < d.n) {
      const double pj = d.p[jj];
      const double qj = st[buf][tid] + (d.h0[jj] + d.sigma[jj]) * pj;
      d.q[jj] = qj;
      pq = fma(pj, qj, pq);
    }
  }
  if (MODE == 0) store_pq_part(d, pq, sh);
}

// Its blocks: as many tiles each as the most loaded block of a resident wave has, on fewer blocks.
static int lr_blocks(const Dev& d, const Geo& g) {
  const int64_t tiles = (d.n + kLrTile - 1) / kLrTile, each = (tiles + g.gN64 - 1) / g.gN64;
  return (int)((tiles + each - 1) / each);
}

static void launch_op_cols(const Dev& d, const Geo& g, int mode, cudaStream_t st) {
  if (lr_alone(d)) {
    const int gl = lr_blocks(d, g);
    if (mode == 0) k_op_cols_lr<0><<<gl, kBlock, 0, st>>>(d);
    else k_op_cols_lr<1><<<gl, kBlock, 0, st>>>(d);
  } else if (d.Hs_ptr || d.ucols || d.aug) {
    if (mode == 0) DISPATCH_G(d.g_cols, k_op_cols<0, G, true><<<g.gN64, kBlock, 0, st>>>(d));
    else if (mode == 1) DISPATCH_G(d.g_cols, k_op_cols<1, G, true><<<g.gN64, kBlock, 0, st>>>(d));
    else DISPATCH_G(d.g_cols, k_op_cols<2, G, true><<<g.gN64, kBlock, 0, st>>>(d));
  } else {
    if (mode == 0) DISPATCH_G(d.g_cols, k_op_cols<0, G, false><<<g.gN64, kBlock, 0, st>>>(d));
    else if (mode == 1) DISPATCH_G(d.g_cols, k_op_cols<1, G, false><<<g.gN64, kBlock, 0, st>>>(d));
    else DISPATCH_G(d.g_cols, k_op_cols<2, G, false><<<g.gN64, kBlock, 0, st>>>(d));
  }
}

// The whole-chip form of the iteration's vector half (pcg.cu's cluster kernel where that does
// not run: BLOCK32 and DENSE preconditioners, systems beyond its size, batches of many solves).
// alpha = rz / p^T q (npart block parts); dx += alpha p; r -= alpha q; ||r||^2 -> convergence test.
// ZM 0 (Jacobi): z = r / M, r^T z, beta.  ZM 1 (Jacobi + low rank): z0 = r / M only.
// ZM 2 (dense): z is left to the dense apply.
template <int ZM>
__global__ void __launch_bounds__(256) k_cg_update(Dev d, int npart) {
  __shared__ double sm[ZM == 0 ? 2 * kBlock : 1];
  __shared__ double sh[32];
  __shared__ double s_alpha;
  Scal* sc = d.sc;
  if (sc->cg_done) return;
  double pq;
  if (ZM == 0) {
    double t1[1] = {0.0}, pq1[1];
    for (int b = threadIdx.x; b < npart; b += blockDim.x) t1[0] += __ldcg(d.partials + 16 * kMaxRedBlocks + b);
    block_sums<1>(t1, sm, pq1);
    pq = pq1[0];
  } else {
    pq = sum_pq_parts(d, npart, sh);   // the cluster kernel's order: either form gives the same bits
  }
  const bool good = pq > 0.0 && isfinite(pq);      // else breakdown: keep the last iterate
  if (threadIdx.x == 0) s_alpha = good ? sc->rz / pq : 0.0;
  __syncthreads();
  const double alpha = s_alpha;
  double rr = 0.0, rz = 0.0;
  if (good)
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.nsys; j += (int64_t)gridDim.x * blockDim.x) {
      d.dx[j] = fma(alpha, d.p[j], d.dx[j]);
      const double rj = fma(-alpha, d.q[j], d.r[j]);
      d.r[j] = rj;
      rr = fma(rj, rj, rr);
      if (ZM < 2) {
        const double zj = rj * d.Minv[j];
        d.z[j] = zj;
        if (ZM == 0) rz = fma(rj, zj, rz);
      }
    }
  if (ZM == 0) {
    // the parts of both sums are added up by every block of k_cg_dir, the next kernel
    const double v[2] = {rr, rz};
    double out[2];
    block_sums<2>(v, sm, out);
    if (threadIdx.x == 0) {
      d.partials[17 * kMaxRedBlocks + blockIdx.x] = out[0];
      d.partials[18 * kMaxRedBlocks + blockIdx.x] = out[1];
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      sc->pq = pq;
      sc->alpha = alpha;
      if (good) {
        sc->cg_iter += 1;
        sc->rz_old = sc->rz;
      } else {
        sc->cg_done = 1;
        if (!isfinite(pq)) sc->status = DS_NUMERICAL;
      }
    }
    return;
  }
  const double v[1] = {rr};
  double out[1];
  if (grid_reduce<1>(v, d.partials + 17 * kMaxRedBlocks, &sc->ticket[T_UPD], out, sh)) {
    if (threadIdx.x == 0) {
      sc->pq = pq;
      sc->alpha = alpha;
      if (!good) {
        sc->cg_done = 1;
        if (!isfinite(pq)) sc->status = DS_NUMERICAL;
        return;
      }
      sc->cg_iter += 1;
      sc->rr = out[0];
      if (!isfinite(out[0])) {
        sc->cg_done = 1;
        sc->status = DS_NUMERICAL;
      } else if (out[0] <= sc->tol2) {
        sc->cg_done = 1;
        sc->cg_conv = 1;
      } else if (sc->cg_iter >= sc->cg_max) {
        sc->cg_done = 1;
      }
    }
  }
}

// After k_cg_update<0>: ||r||^2 and r^T z from its parts, the test, beta, and the next direction.
// Every block adds up the parts and comes to the same decision; block 0 writes the scalars that
// no other block reads here (n = 77373: 13.0 us for the two kernels; 16.4 us with a last-block
// reduction and three shuffle trees in all warps of k_cg_update).
__global__ void __launch_bounds__(256) k_cg_dir(Dev d, int npart, cudaGraphConditionalHandle h, int set_cond) {
  __shared__ double sm[2 * kBlock];
  __shared__ double s_beta;
  Scal* sc = d.sc;
  const bool first = blockIdx.x == 0 && threadIdx.x == 0;
  if (sc->cg_done) {
    if (set_cond && first) cudaGraphSetConditional(h, 0u);
    return;
  }
  double v[2] = {0.0, 0.0}, out[2];
  for (int b = threadIdx.x; b < npart; b += blockDim.x) {
    v[0] += __ldcg(d.partials + 17 * kMaxRedBlocks + b);
    v[1] += __ldcg(d.partials + 18 * kMaxRedBlocks + b);
  }
  block_sums<2>(v, sm, out);
  const bool bad = !isfinite(out[0]), conv = out[0] <= sc->tol2;
  const bool done = bad || conv || sc->cg_iter >= sc->cg_max;
  if (threadIdx.x == 0) s_beta = out[1] / sc->rz_old;
  __syncthreads();
  const double beta = s_beta;
  if (!done)
    for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.nsys; j += (int64_t)gridDim.x * blockDim.x) {
      const double pj = fma(beta, d.p[j], d.z[j]);
      d.p[j] = pj;
      if (d.p32) d.p32[j] = (float)pj;
      if (d.p_df && j < d.n) d.p_df[j] = df_split(pj);
    }
  if (first) {
    if (set_cond) cudaGraphSetConditional(h, done ? 0u : 1u);
    sc->rr = out[0];
    if (bad) sc->status = DS_NUMERICAL;
    if (!bad && conv) sc->cg_conv = 1;
    if (done) {
      sc->cg_done = 1;
    } else {
      sc->beta = beta;
      sc->rz = out[1];
    }
  }
}

// Low-rank correction (Woodbury): with z0 = M^{-1} r already in z,
//   z = z0 - M^{-1} A_s^T G^{-1} A_s z0.
// k_stiff_u: u_a = A_s z0 (one warp per stiff row).
__global__ void k_stiff_u(Dev d, int init) {
  if (!init && d.sc->cg_done) return;
  const int ns = d.sc->n_stiff;
  for (int a = gwarp(); a < ns; a += nwarps()) {
    const int32_t row = d.arow[d.stiff_k[a]];
    double u = warp_row_dot<false>(d.R_ptr[row], d.R_ptr[row + 1], d.R_idx, d.R_val, d.z);
    if ((threadIdx.x & 31) == 0) d.us[a] = u;
  }
}

// t = G^{-1} u (dense symmetric matvec, one warp per output).
__global__ void k_stiff_t(Dev d, int init) {
  if (!init && d.sc->cg_done) return;
  const int ns = d.sc->n_stiff;
  const int cap = d.stiff_cap;
  const int lane = threadIdx.x & 31;
  for (int a = gwarp(); a < ns; a += nwarps()) {
    const double* g = d.Ginv + (int64_t)a * cap;
    double acc = 0.0;
    for (int b = lane; b < ns; b += 32) acc = fma(g[b], d.us[b], acc);
    acc = warp_sum(acc);
    if (lane == 0) d.ts[a] = acc;
  }
}

// z_j = z0_j - Minv_j sum_{(a, v) in column j} v t_a; r^T z -> beta (loop) or rz (init);
// in init mode also p = z.
__global__ void k_stiff_corr(Dev d, int init) {
  __shared__ double sh[32];
  if (!init && d.sc->cg_done) return;
  const int ns = d.sc->n_stiff;
  double rz = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * blockDim.x) {
    double zj = d.z[j];
    if (ns > 0) {
      double acc = 0.0;
      const int2 run = d.sc_run[j];
      for (int t = run.x; t < run.x + run.y; ++t) acc = fma(d.sc_val[t], d.ts[d.sc_slot[t]], acc);
      zj -= d.Minv[j] * acc;
      d.z[j] = zj;
    }
    if (init) {
      d.p[j] = zj;
      if (d.p32) d.p32[j] = (float)zj;
      if (d.p_df) d.p_df[j] = df_split(zj);
    }
    rz = fma(d.r[j], zj, rz);
  }
  double v[1] = {rz};
  double out[1];
  if (grid_reduce<1>(v, d.partials + 19 * kMaxRedBlocks, &d.sc->ticket[T_CORR], out, sh)) {
    if (threadIdx.x == 0) {
      Scal* sc = d.sc;
      if (init) {
        sc->rz = out[0];
      } else {
        sc->beta = out[0] / sc->rz;
        sc->rz = out[0];
      }
    }
  }
}

// Dense preconditioner apply by triangular solves in double-float pairs: z = K^{-1} r with
// s K = L L^T (the scaled K factored in pairs: L in the lower triangle of Kd, L^T mirrored
// into the upper triangle, both row-major), forward L y = r' then backward L^T z' = y, where
// r' = 2^-e r (2^e >= max |r|, exact) and z = s 2^e z'.  In blocks of 32 rows: the block's
// 32 values come from the inverse of its diagonal tile (one warp per row, a shuffle-tree sum
// of pairs: no row-by-row chain), then all threads update the remaining rows with the block's
// 32 columns.  One block of 1024 threads; y in shared memory (n <= 2048).  r^T z -> rz / beta;
// init: p = z.  (PCG with the factor converges in one or two iterations, so this replaces
// forming K^{-1} once per IPM iteration.)
//
// The chain of 2 n / 32 steps is what bounds it, so nothing in a step waits for memory that
// could have been asked for before: each thread pair's 32 factor entries of the next block (16
// entries a thread, in 16-byte loads where rows start on 16 bytes) and the next tile's inverse
// are fetched into registers before the barriers of the current step, and a row's 32 terms are
// split over two threads with two accumulators each.  (n = 500: 128 us for the two sweeps with one
// thread a row loading as it went.)
struct TrsvRow {
  float2 v[16];
};
// 16 entries of a row from column c0; VEC: 16-byte loads (row and column even)
template <bool VEC>
__device__ __forceinline__ void trsv_fetch(const float2* row, int c0, int left, TrsvRow& t) {
  if (VEC && left >= 16) {
    const float4* p = reinterpret_cast<const float4*>(row + c0);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const float4 u = p[k];
      t.v[2 * k] = make_float2(u.x, u.y);
      t.v[2 * k + 1] = make_float2(u.z, u.w);
    }
  } else {
#pragma unroll
    for (int k = 0; k < 16; ++k) t.v[k] = k < left ? row[c0 + k] : make_float2(0.f, 0.f);
  }
}
__device__ __forceinline__ void trsv_dot(const TrsvRow& t, const float2* yk, float& h, float& l) {
  float h0 = 0.f, l0 = 0.f, h1 = 0.f, l1 = 0.f;
#pragma unroll
  for (int k = 0; k < 16; k += 2) {
    df_mac(t.v[k], yk[k], h0, l0);
    df_mac(t.v[k + 1], yk[k + 1], h1, l1);
  }
  float e;
  two_sum(h0, h1, h, e);
  l = __fadd_rn(__fadd_rn(l0, l1), e);
}

// y[r] -= row r's 32 terms for rows r0 <= r < r1 (rows beyond the first 512 of the range load as
// they go), two neighbouring threads a row; `row`: the thread's fetched part of row r0 + tid / 2.
template <bool VEC>
__device__ __forceinline__ void trsv_rows(const float2* K, int64_t ld, int kb, int bs, int r0, int r1, float2* y,
                                          const float2* yk, TrsvRow& row) {
  const int tid = threadIdx.x, half = tid & 1, c0 = 16 * half;
  for (int rr = r0; rr < r1; rr += 512) {
    const int r = rr + (tid >> 1);
    if (rr != r0 && r < r1) trsv_fetch<VEC>(K + (int64_t)r * ld, kb + c0, bs - c0, row);
    float h = 0.f, l = 0.f;
    if (r < r1) trsv_dot(row, yk + c0, h, l);
    const float oh = __shfl_xor_sync(0xffffffffu, h, 1), ol = __shfl_xor_sync(0xffffffffu, l, 1);
    if (r < r1 && half == 0) {
      float sm, e;
      two_sum(h, oh, sm, e);
      y[r] = df_sub_sum(y[r], sm, __fadd_rn(__fadd_rn(l, ol), e));
    }
  }
}

template <bool VEC>
__global__ void __launch_bounds__(1024) k_dense_trsv(Dev d, int init) {
  extern __shared__ float2 y[];
  __shared__ double sh[32];
  __shared__ float2 Li[32][33];
  __shared__ float2 yk[32];
  if (!init && d.sc->cg_done) return;
  const int n = (int)d.n;
  const int nt = (n + 31) / 32;
  const float2* K = d.Kd;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, c0 = 16 * (tid & 1);
  // tile t's inverse entry and the thread's part of its row below (forward) or above (backward)
  // the tile, for the step to come
  float2 li = d.chol_tinv[warp * 32 + lane];
  TrsvRow row;
  auto fetch_fwd = [&](int t) {
    const int kb = t * 32, bs = min(32, n - kb), r = kb + bs + (tid >> 1);
    if (r < n) trsv_fetch<VEC>(K + (int64_t)r * n, kb + c0, bs - c0, row);
  };
  auto fetch_bwd = [&](int t) {
    const int kb = t * 32, bs = min(32, n - kb), r = tid >> 1;
    if (r < kb) trsv_fetch<VEC>(K + (int64_t)r * n, kb + c0, bs - c0, row);
  };
  fetch_fwd(0);
  double rmax = 0.0;
  for (int i = tid; i < n; i += blockDim.x) rmax = fmax(rmax, fabs(d.r[i]));
  rmax = block_reduce<1>(rmax, sh);
  int er = 0;
  if (rmax > 0.0 && isfinite(rmax)) frexp(rmax, &er);
  const double rs = ldexp(1.0, -er);
  for (int i = tid; i < n; i += blockDim.x) y[i] = df_split(d.r[i] * rs);
  Li[warp][lane] = li;
  __syncthreads();
  // forward: L y = r'
  for (int t = 0; t < nt; ++t) {
    const int kb = t * 32, bs = min(32, n - kb);
    if (t + 1 < nt) li = d.chol_tinv[(int64_t)(t + 1) * 1024 + warp * 32 + lane];
    float h = 0.f, l = 0.f;
    if (lane < bs) df_mac(Li[warp][lane], y[kb + lane], h, l);
    df_group_pair<32>(h, l);
    if (lane == 0) yk[warp] = df_fast_sum(h, l);
    __syncthreads();
    if (tid < bs) y[kb + tid] = yk[tid];
    trsv_rows<VEC>(K, n, kb, bs, kb + bs, n, y, yk, row);
    if (t + 1 < nt) {
      Li[warp][lane] = li;
      fetch_fwd(t + 1);
    } else {
      fetch_bwd(t);
    }
    __syncthreads();
  }
  // backward: L^T z' = y, with L^T row i in the upper triangle of row i; tile nt - 1's
  // inverse is still staged
  for (int t = nt - 1; t >= 0; --t) {
    const int kb = t * 32, bs = min(32, n - kb);
    if (t > 0) li = d.chol_tinv[(int64_t)(t - 1) * 1024 + warp * 32 + lane];
    float h = 0.f, l = 0.f;
    if (lane < bs) df_mac(Li[lane][warp], y[kb + lane], h, l);
    df_group_pair<32>(h, l);
    if (lane == 0) yk[warp] = df_fast_sum(h, l);
    __syncthreads();
    if (tid < bs) y[kb + tid] = yk[tid];
    trsv_rows<VEC>(K, n, kb, bs, 0, kb, y, yk, row);
    if (t > 0) {
      Li[warp][lane] = li;
      fetch_bwd(t - 1);
    }
    __syncthreads();
  }
  const double zs = d.dense_aux[2] * ldexp(1.0, er);
  double rz = 0.0;
  for (int j = tid; j < n; j += blockDim.x) {
    const double zj = df_value(y[j].x, y[j].y) * zs;
    d.z[j] = zj;
    if (init) {
      d.p[j] = zj;
      if (d.p32) d.p32[j] = (float)zj;
      if (d.p_df) d.p_df[j] = df_split(zj);
    }
    rz = fma(d.r[j], zj, rz);
  }
  rz = block_reduce<0>(rz, sh);
  if (tid == 0) {
    Scal* sc = d.sc;
    if (init) {
      sc->rz = rz;
    } else {
      sc->beta = rz / sc->rz;
      sc->rz = rz;
    }
  }
}

static void launch_trsv(const Dev& d, int init, cudaStream_t st) {
  if (d.n & 1) k_dense_trsv<false><<<1, 1024, sizeof(float2) * d.n, st>>>(d, init);
  else k_dense_trsv<true><<<1, 1024, sizeof(float2) * d.n, st>>>(d, init);
}

// Jacobi start: z = r / M, p = z, rz = r^T z.
__global__ void k_cg_init_diag(Dev d) {
  __shared__ double sh[32];
  double rz = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.nsys; j += (int64_t)gridDim.x * blockDim.x) {
    const double zj = d.r[j] * d.Minv[j];
    d.z[j] = zj;
    d.p[j] = zj;
    if (d.p32) d.p32[j] = (float)zj;
    if (d.p_df && j < d.n) d.p_df[j] = df_split(zj);
    rz = fma(d.r[j], zj, rz);
  }
  double v[1] = {rz};
  double out[1];
  if (grid_reduce<1>(v, d.partials + 21 * kMaxRedBlocks, &d.sc->ticket[T_CORR], out, sh)) {
    if (threadIdx.x == 0) d.sc->rz = out[0];
  }
}

// p = z + beta p; also sets the while-loop condition of the captured PCG graph.
__global__ void k_cg_p(Dev d, cudaGraphConditionalHandle h, int set_cond) {
  const int done = d.sc->cg_done;
  if (set_cond && blockIdx.x == 0 && threadIdx.x == 0) cudaGraphSetConditional(h, done ? 0u : 1u);
  if (done) return;
  const double beta = d.sc->beta;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.nsys; j += (int64_t)gridDim.x * blockDim.x)
  {
    const double pj = fma(beta, d.p[j], d.z[j]);
    d.p[j] = pj;
    if (d.p32) d.p32[j] = (float)pj;
    if (d.p_df && j < d.n) d.p_df[j] = df_split(pj);
  }
}

cudaError_t launch_cg_init(const Dev& d, const Geo& g, int precond, cudaStream_t st, cudaGraphConditionalHandle h) {
  if (tail_runs(d, precond)) return launch_tail_init(d, precond, h, st);
  if (h) {
    const cudaError_t e = launch_set_cond(h, 1u, st);
    if (e != cudaSuccess) return e;
  }
  if (precond == PC_BLOCK32) return launch_block_apply(d, 1, st);
  if (precond == PC_DENSE) {
    launch_trsv(d, 1, st);
  } else {
    k_cg_init_diag<<<g.eN, kBlock, 0, st>>>(d);
    if (precond == PC_JACOBI_LR && d.m) {
      const int gs = (d.stiff_cap + 7) / 8;
      k_stiff_u<<<gs, kBlock, 0, st>>>(d, 1);
      k_stiff_t<<<gs, kBlock, 0, st>>>(d, 1);
      k_stiff_corr<<<g.eN, kBlock, 0, st>>>(d, 1);
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_cg_body(const Dev& d, const Geo& g, int precond, cudaGraphConditionalHandle h, cudaStream_t st,
                           bool in_graph, bool lowp) {
  const bool tail = tail_runs(d, precond);
  // one block an SM: every block adds up the parts of p^T q and one more tree of partial sums (the
  // reduced storages keep the blocks their results are rounded by)
  const int gU = d.storage == ST_F64 ? std::min(g.eN, d.sm_count > 0 ? d.sm_count : 148) : g.eN;
  int npart = g.gNc;
  if (lowp) {
    cudaError_t e = launch_op_lp(d, g, !tail, st);
    if (e != cudaSuccess) return e;
  } else if (d.mx) {
    launch_op_rows_mx(d, g, 0, st);
    launch_lr(d, d.p, 0, st);
    launch_op_cols_mx(d, g, 0, st);
  } else if (d.df) {
    launch_op_rows_df(d, g, 0, st);
    launch_lr(d, d.p, 0, st);
    launch_op_cols_df(d, g, 0, st);
  } else {
    if (d.runs) launch_op_rows_runs(d, g, 0, st);
    else if (d.nR) DISPATCH_G(d.g_rows, k_op_rows<0, G><<<g.gR64, kBlock, 0, st>>>(d));
    launch_lr(d, d.p, 0, st);
    launch_op_cols(d, g, 0, st);
    npart = lr_alone(d) ? lr_blocks(d, g) : g.gN64;
  }
  if (tail) return launch_tail_iter(d, precond, npart, h, in_graph, st);
  if (precond == PC_BLOCK32) {
    k_cg_update<2><<<gU, kBlock, 0, st>>>(d, npart);
    launch_block_apply(d, 0, st);
  } else if (precond == PC_DENSE) {
    k_cg_update<2><<<gU, kBlock, 0, st>>>(d, npart);
    launch_trsv(d, 0, st);
  } else if (precond == PC_JACOBI_LR && d.m) {
    k_cg_update<1><<<gU, kBlock, 0, st>>>(d, npart);
    const int gs = (d.stiff_cap + 7) / 8;
    k_stiff_u<<<gs, kBlock, 0, st>>>(d, 0);
    k_stiff_t<<<gs, kBlock, 0, st>>>(d, 0);
    k_stiff_corr<<<g.eN, kBlock, 0, st>>>(d, 0);
  } else if (d.crowd && !d.aug) {
    // in a crowded batch for the cluster kernel: its order of r^T z, so its bits (no stiff rows here)
    k_cg_update<1><<<gU, kBlock, 0, st>>>(d, npart);
    k_stiff_corr<<<g.eN, kBlock, 0, st>>>(d, 0);
  } else {
    k_cg_update<0><<<gU, kBlock, 0, st>>>(d, npart);
    k_cg_dir<<<gU, kBlock, 0, st>>>(d, gU, h, in_graph ? 1 : 0);
    return cudaGetLastError();
  }
  k_cg_p<<<g.eN, kBlock, 0, st>>>(d, h, in_graph ? 1 : 0);
  return cudaGetLastError();
}

// The rows and the column pass of the handle's FP64-storage PCG operator alone (measurement,
// autotuning); the double-float passes read p_df, which the caller keeps current.
// The low-rank correction of the preconditioner after z0 = r / M (loop form) and the next
// search direction (with the loop condition), for the replacement PCG of lowp.cu.
cudaError_t launch_stiff_apply(const Dev& d, const Geo& g, cudaStream_t st) {
  const int gs = (d.stiff_cap + 7) / 8;
  k_stiff_u<<<gs, kBlock, 0, st>>>(d, 0);
  k_stiff_t<<<gs, kBlock, 0, st>>>(d, 0);
  k_stiff_corr<<<g.eN, kBlock, 0, st>>>(d, 0);
  return cudaGetLastError();
}

cudaError_t launch_cg_p(const Dev& d, const Geo& g, cudaGraphConditionalHandle h, bool in_graph, cudaStream_t st) {
  k_cg_p<<<g.eN, kBlock, 0, st>>>(d, h, in_graph ? 1 : 0);
  return cudaGetLastError();
}

cudaError_t launch_op_rows_only(const Dev& d, const Geo& g, cudaStream_t st) {
  if (d.mx) return launch_op_rows_mx(d, g, 1, st);
  if (d.df) return launch_op_rows_df(d, g, 1, st);
  if (d.runs) return launch_op_rows_runs(d, g, 1, st);
  if (d.nR) DISPATCH_G(d.g_rows, k_op_rows<1, G><<<g.gR64, kBlock, 0, st>>>(d));
  return cudaGetLastError();
}

cudaError_t launch_op_cols_only(const Dev& d, const Geo& g, cudaStream_t st) {
  // (the low-rank term uses us from the last launch_lr; the measurement does not re-run it)
  if (d.mx) return launch_op_cols_mx(d, g, 1, st);
  if (d.df) return launch_op_cols_df(d, g, 1, st);
  launch_op_cols(d, g, 1, st);
  return cudaGetLastError();
}

// q = K p, one apply of the handle's FP64-storage PCG operator (FP64 or double-float).
cudaError_t launch_apply(const Dev& d, const Geo& g, cudaStream_t st) {
  if (d.mx) {
    launch_mirror_df(d, g, st);
    launch_op_rows_mx(d, g, 1, st);
    launch_lr(d, d.p, 0, st);
    launch_op_cols_mx(d, g, 1, st);
    return cudaGetLastError();
  }
  if (d.df) {
    launch_mirror_df(d, g, st);
    launch_op_rows_df(d, g, 1, st);
    launch_lr(d, d.p, 0, st);
    launch_op_cols_df(d, g, 1, st);
    return cudaGetLastError();
  }
  // (a reduced-storage handle keeps runs for its narrow rows pass; its FP64 applies read CSR,
  // the faster FP64 form)
  if (d.runs && d.storage == ST_F64) launch_op_rows_runs(d, g, 1, st);
  else if (d.nR) DISPATCH_G(d.g_rows, k_op_rows<1, G><<<g.gR64, kBlock, 0, st>>>(d));
  launch_lr(d, d.p, 0, st);
  launch_op_cols(d, g, 1, st);
  return cudaGetLastError();
}

// q = K dx when the reduced-precision PCG asks for a residual replacement (ru_do), else
// nothing: the FP64 operator over the accumulated step (a copy of the bundle with p -> dx).
cudaError_t launch_apply_ru(const Dev& d, const Geo& g, cudaStream_t st) {
  Dev d2 = d;
  d2.p = d.dx;
  if (d.nR) DISPATCH_G(d.g_rows, k_op_rows<2, G><<<g.gR64, kBlock, 0, st>>>(d2));
  if (d.ucols) launch_lr(d2, d2.p, 0, st);
  launch_op_cols(d2, g, 2, st);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ recovery

// The ratio test's quotient -v / dv of a v that falls (INFINITY otherwise), as the key that orders
// quotients on the integer pipe: block and grid minima run there, with one atomic a warp, and come
// out as fmin's would (NaN is passed over; a negative quotient, of a v that rounding put past its
// bound, counts as the number it is).
__device__ __forceinline__ void keep_ratio(long long& m, double v, double dv) {
  if (dv < 0.0) {
    const long long k = min_key(__double_as_longlong(-v / dv));
    m = k < m ? k : m;
  }
}

// Minima of a block into the step's (primal, dual).
__device__ __forceinline__ void block_ratio(const Dev& d, long long ap, long long ad) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long a = __shfl_xor_sync(0xffffffffu, ap, o), b = __shfl_xor_sync(0xffffffffu, ad, o);
    ap = a < ap ? a : ap;
    ad = b < ad ? b : ad;
  }
  if ((threadIdx.x & 31) == 0) {
    if (ap < kInfBits) atomicMin(&d.sc->step_min[0], ap);
    if (ad < kInfBits) atomicMin(&d.sc->step_min[1], ad);
  }
}

// alpha = min(1, tau times the minimum ratio), separate for (x, s) and (y, z) or their minimum.
__device__ __forceinline__ void step_lengths(const Scal* sc, double& a_p, double& a_d) {
  a_p = fmin(1.0, sc->tau * __longlong_as_double(min_key_bits(sc->step_min[0])));
  a_d = fmin(1.0, sc->tau * __longlong_as_double(min_key_bits(sc->step_min[1])));
  if (sc->equal_steps) a_p = a_d = fmin(a_p, a_d);
}

// The full direction and its ratio test in one launch.  Blocks [0, gm): constraint rows, A dx by
// groups of G lanes, then ds = -r_p - A dx and dy = theta (A dx + r_p) - r_s / s by the block's
// first 256 / G threads (as in k_cols_resid); the other blocks: dz_l = (-r_l - z_l dx) / t_l,
// dz_u = (-r_u + z_u dx) / t_u.  (Five launches before, 29 us at n = 7001.)
template <int G>
__global__ void k_recover(Dev d, int gm) {
  constexpr int C = kBlock / G;
  __shared__ double st[2][C];
  const double mu = d.sc->mu;
  long long ap = kInfBits, ad = kInfBits;
  const int tid = threadIdx.x;
  if ((int)blockIdx.x < gm) {
    int buf = 0;
    for (int64_t k0 = (int64_t)blockIdx.x * C; k0 < d.m; k0 += (int64_t)gm * C, buf ^= 1) {
      const int64_t kg = k0 + tid / G;
      const bool ok = kg < d.m;
      const int32_t row = ok ? d.arow[kg] : 0;
      const int64_t beg = ok ? d.R_ptr[row] : 0, end = ok ? d.R_ptr[row + 1] : 0;
      const double t = group_row_dot<G, false>(beg, end, glane<G>(), d.R_idx, d.R_val, d.dx);
      if (glane<G>() == 0) st[buf][tid / G] = t;
      __syncthreads();
      const int64_t k = k0 + tid;
      if (tid < C && k < d.m) {
        const double adx = st[buf][tid], s = d.s[k], y = d.y[k], rp = d.rp[k];
        const double ds = -rp - adx;
        // doubly augmented: dy is the solved bottom block
        // each operation rounded by itself: the value does not hang on how the compiler would fuse
        const double dy = d.aug ? d.dx[d.n + k]
                                : __dsub_rn(__dmul_rn(d.theta[k], adx + rp), __dsub_rn(__dmul_rn(s, y), mu) / s);
        d.ds[k] = ds;
        d.dy[k] = dy;
        keep_ratio(ap, s, ds);
        keep_ratio(ad, y, dy);
      }
    }
  } else {
    const int64_t nb = (int64_t)gridDim.x - gm;
    for (int64_t j = ((int64_t)blockIdx.x - gm) * blockDim.x + tid; j < d.n; j += nb * blockDim.x) {
      const double xj = d.x[j], dxj = d.dx[j];
      double dzl = 0.0, dzu = 0.0;
      if (d.fl[j]) {
        const double tl = xj - d.l[j], z = d.zl[j];
        const double rl = tl * z - mu;
        dzl = (-rl - z * dxj) / tl;
        keep_ratio(ap, tl, dxj);
        keep_ratio(ad, z, dzl);
      }
      if (d.fu[j]) {
        const double tu = d.u[j] - xj, z = d.zu[j];
        const double ru = tu * z - mu;
        dzu = (-ru + z * dxj) / tu;
        keep_ratio(ap, tu, -dxj);
        keep_ratio(ad, z, dzu);
      }
      d.dzl[j] = dzl;
      d.dzu[j] = dzu;
    }
  }
  block_ratio(d, ap, ad);
}

cudaError_t launch_recover(const Dev& d, const Geo& g, cudaStream_t st) {
  DISPATCH_G(d.g_rows, k_recover<G><<<g.gM + g.eN, kBlock, 0, st>>>(d, g.gM));
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ ratio test

// The ratio test alone, on given directions (the step-level call).
__global__ void k_ratio_begin(Dev d) {
  if (threadIdx.x < 2) d.sc->step_min[threadIdx.x] = kInfBits;
}

__global__ void k_ratio(Dev d) {
  long long ap = kInfBits, ad = kInfBits;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x) {
    keep_ratio(ap, d.s[k], d.ds[k]);
    keep_ratio(ad, d.y[k], d.dy[k]);
  }
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * blockDim.x) {
    const double xj = d.x[j], dxj = d.dx[j];
    if (d.fl[j]) { keep_ratio(ap, xj - d.l[j], dxj); keep_ratio(ad, d.zl[j], d.dzl[j]); }
    if (d.fu[j]) { keep_ratio(ap, d.u[j] - xj, -dxj); keep_ratio(ad, d.zu[j], d.dzu[j]); }
  }
  block_ratio(d, ap, ad);
}

__global__ void k_ratio_end(Dev d) {
  if (threadIdx.x == 0) {
    double a_p, a_d;
    step_lengths(d.sc, a_p, a_d);
    d.sc->alpha_p = a_p;
    d.sc->alpha_d = a_d;
  }
}

cudaError_t launch_ratio(const Dev& d, const Geo& g, cudaStream_t st) {
  k_ratio_begin<<<1, 32, 0, st>>>(d);
  k_ratio<<<std::max(g.eN, g.eM), kBlock, 0, st>>>(d);
  k_ratio_end<<<1, 32, 0, st>>>(d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ update

// x, s by alpha_p, y, z by alpha_d; one thread a block forms the step lengths.
__global__ void k_update(Dev d) {
  __shared__ double al[2];
  if (threadIdx.x == 0) {
    step_lengths(d.sc, al[0], al[1]);
    if (blockIdx.x == 0) {
      d.sc->alpha_p = al[0];
      d.sc->alpha_d = al[1];
    }
  }
  __syncthreads();
  const double ap = al[0], ad = al[1];
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < d.n; j += (int64_t)gridDim.x * blockDim.x) {
    d.x[j] = fma(ap, d.dx[j], d.x[j]);
    if (d.fl[j]) d.zl[j] = fma(ad, d.dzl[j], d.zl[j]);
    if (d.fu[j]) d.zu[j] = fma(ad, d.dzu[j], d.zu[j]);
  }
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < d.m; k += (int64_t)gridDim.x * blockDim.x) {
    d.s[k] = fma(ap, d.ds[k], d.s[k]);
    d.y[k] = fma(ad, d.dy[k], d.y[k]);
  }
}

cudaError_t launch_update(const Dev& d, const Geo& g, cudaStream_t st) {
  k_update<<<std::max(g.eN, g.eM), kBlock, 0, st>>>(d);
  return cudaGetLastError();
}

// ------------------------------------------------------------------------------ precond build

cudaError_t launch_dense_build(const Dev& d, cudaStream_t st);       // dense.cu
cudaError_t launch_stiff_factor(const Dev& d, cudaStream_t st);      // dense.cu

cudaError_t prepare_steps() {
  cudaError_t e = cudaFuncSetAttribute(k_gram_G, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       kGramSlots * 8 * kGramEntries * 6);
  // Shared memory (percent) for two blocks an SM, not for all that fit: an SM changes its split of
  // L1 and shared memory only when idle, so beside other solves the split of one kernel stays for
  // all, and the operator passes live on their L1 (64 QPs in one launch: 49.0 solves/s with the
  // default, 62.5 with one block's share, 63.1 with two; alone one block's share costs 4 us in 15).
  constexpr int kGramCarveout = 44;
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_gram_G, cudaFuncAttributePreferredSharedMemoryCarveout, kGramCarveout);
  return e;
}

// Before the right-hand side: stiff-row selection (JACOBI_LR).
cudaError_t launch_precond_build(const Dev& d, const Geo& g, int precond, cudaStream_t st) {
  if (precond == PC_JACOBI_LR && d.m) DISPATCH_G(d.g_rows, k_stiff_select<G><<<g.gM, kBlock, 0, st>>>(d));
  return cudaGetLastError();
}

// After the right-hand side (which also wrote the Jacobi diagonal): the low-rank factor
// (JACOBI_LR) or the dense factor (DENSE).
cudaError_t launch_precond_finish(const Dev& d, const Geo& g, int precond, cudaStream_t st) {
  if (precond == PC_DENSE) return launch_dense_build(d, st);
  if (precond == PC_BLOCK32) return launch_block_factor(d, st);
  if (precond == PC_JACOBI_LR && d.m) {
    const int nb = (d.stiff_cap + 7) / 8;
    k_sc_mask<<<nb, kBlock, 0, st>>>(d);
    k_sc_runs<<<g.eN, kBlock, 0, st>>>(d);
    k_sc_fill<<<nb, kBlock, 0, st>>>(d);
    k_gram_G<<<d.stiff_cap, 256, (size_t)d.sc_words * kGramEntries * 6, st>>>(d);
    cudaError_t e = launch_stiff_factor(d, st);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

}  // namespace ipmk
