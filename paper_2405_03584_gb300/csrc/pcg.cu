// The vector half of a PCG iteration in one kernel (sm_103a): everything between the column
// pass of the operator (q = K p) and the next rows pass.
//
//   alpha = rz / p^T q;  dx += alpha p;  r -= alpha q;  ||r||^2 and the convergence test;
//   z = P^{-1} r (Jacobi, or Jacobi with the stiff rows' low-rank correction);
//   beta = r^T z / rz;  p = z + beta p  (and the narrow mirrors of p);
//   reduced storage: the exact FP64 product of the stiff rows with the new p.
//
// What bounds it: latency, and the float64 pipe.  The vectors are a few hundred KB; a global
// sum is a synchronisation of every thread; and GB300 gives each quarter of an SM half a
// float64 lane a clock, so every float64 warp instruction holds its quarter for 64 cycles,
// however many lanes it serves: an instruction that every warp of a block executes for a value
// they all share costs more than a barrier.  As separate kernels (update, A_s z, G^{-1} u,
// correction, p), each with its own last-block sum, the half took 27 us an iteration at n =
// 1500 and 34 us at n = 50000 (9 us and 22 us here).  One thread-block cluster runs it
// instead: its CTAs are resident together, so a global sum is one exchange through distributed
// shared memory and one cluster barrier, the vectors stay in registers from the update to the
// new p, and the loads of a phase are issued before the barrier that precedes it.  Scalars are
// formed by one warp and handed out through shared memory; warps without unknowns skip the vector arithmetic; the trees of a
// sum are formed from shared memory by 8 lanes per 32 values (6 float64 instructions for four
// trees a warp, against 20 by shuffles alone).
//
// Every sum that feeds the iteration (p^T q, r^T z, the stiff rows' products) has one fixed order
// (blocks of 256 values as warp trees, then the blocks' parts as one such block) for every shape
// of the cluster, so the shape does not show in the result, bit for bit; only ||r||^2, which is
// compared with tolerances alone, is added in an order of its own.
//
// One cluster of 16 SMs streams about 2 TB/s and has a tenth of the chip's float64 rate, so
// the kernel stops paying where the vectors outgrow it: above kTailMaxN unknowns (kTailPlainN
// without the stiff rows' correction), and where the device has no room for such a cluster,
// tail_runs() declines and the caller takes the whole-chip kernels.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "state.h"

namespace ipmk {

namespace {

constexpr int kTailThreads = 512;
constexpr int kTailWarps = kTailThreads / 32;
constexpr int kTailCtas = 16;          // CTAs of the largest cluster (16 needs the non-portable opt-in)
constexpr int64_t kTailSmall = 512;    // unknowns up to which the cluster has 8 CTAs
constexpr int kTailMaxE = 7;           // unknowns per thread
constexpr int64_t kTailMaxN = (int64_t)kTailCtas * kTailThreads * kTailMaxE;
// Without the stiff rows' correction the whole-chip form is two kernels, and the shorter one from
// about 20000 unknowns on: whole solves with H's low-rank term alone take 3.33 ms by the cluster
// and 3.43 by the chip at n = 16384, 3.54 and 3.44 at 24000, 3.92 and 3.68 at 45000 (with the
// correction it is five, and the cluster the shorter one at every size it holds).  The reduced
// storages stay with the cluster: their results are rounded by its sums.
constexpr int64_t kTailPlainN = (int64_t)kTailCtas * kTailThreads * 2;
constexpr int kStiffCapMax = 1024;     // options.stiff_max's limit
constexpr int kPre = 8;                // entries per lane fetched before a barrier

enum TailMode { TAIL_ITER = 0, TAIL_INIT = 1, TAIL_RU = 2, TAIL_RU2 = 3 };

__device__ __forceinline__ void cl_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cl_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

// v into the double at `p` (an address of this CTA's shared memory) of CTA `rank`.
__device__ __forceinline__ void cl_store(const double* p, int rank, double v) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}

constexpr int kTailBlocks = kTailMaxE * 2 * kTailCtas;   // blocks of 256 unknowns, at most
static_assert(kTailBlocks <= 256, "the last tree takes one block part a thread");

template <int E>
struct TailShared {
  union {
    struct {
      double u[kStiffCapMax], t[kStiffCapMax];
    };
    double red[16 * E * 33];           // 16 E warps of values, 33 apart (no bank conflicts either way)
  };
  double wsum[16 * E];                 // sums of the warps of values
  double rr[16 * 33], rw[16];          // the threads' parts of ||r||^2 and their warps' sums
  double part[kTailBlocks];            // r^T z of every block of 256 unknowns, of all CTAs
  double xrr[kTailCtas];
  double w8[8];
  double alpha, beta, rz;
  int stop;
};

// The sum of up to 8 * 32 values, value i in lane i & 31 of warp i >> 5 (0 beyond), as a block
// of 256 threads sums them: warp trees, then a tree over the warps; result in warp 0 (lane 0).
// nv: values (the same in every thread).
__device__ __forceinline__ double block_tree(double v, int nv, double* w8) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double t = 0.0;
  if (32 * w < nv) t = warp_sum(v);
  if (nv <= 32) return t;
  if (w < 8 && lane == 0) w8[w] = t;
  __syncthreads();
  if (w == 0) {
    t = lane < 8 ? w8[lane] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1)
      if (32 * o < nv) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  return t;
}

// Tree sums (as warp_sum adds them) of cnt runs of 32 values, 33 apart at v, into dst[]: 8 lanes
// a run by the threads of warps w0, w0 + 1, ... of the block, as far as they reach.
__device__ __forceinline__ void tree_runs(const double* v, int cnt, double* dst, int w0) {
  const int lane = threadIdx.x & 31, g = lane & 7;
  for (int b = 4 * ((int)(threadIdx.x >> 5) - w0); b < cnt; b += 4 * (kTailWarps - w0)) {
    const int k = b + (lane >> 3);
    double t = 0.0;
    if (k < cnt) {
      const double* x = v + 33 * k + g;
      t = (x[0] + x[16]) + (x[8] + x[24]);
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (g == 0 && k < cnt) dst[k] = t;
  }
}

// The same by one thread a run: fewer instructions where there are many runs.
__device__ __forceinline__ double tree32(const double* v) {
  double a[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) a[i] = v[i] + v[i + 16];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < o; ++i) a[i] += a[i + o];
  return a[0];
}

__device__ __forceinline__ bool positive_finite(double v) {
  const long long b = __double_as_longlong(v);
  return b > 0 && b < 0x7ff0000000000000ll;
}

// A stiff row's product with a vector by one warp: its first 256 entries are fetched ahead of
// time (stiff_fetch); the vector, which this kernel has written, is read through L2.  Lane l
// adds entries l, l + 32, ... in the order of warp_row_dot: four accumulators while four whole
// strides remain, the rest into the first.
struct StiffRow {
  int64_t beg;
  int len;
  double v[kPre];
  int i[kPre];
};

__device__ __forceinline__ void stiff_range(const Dev& d, int a, int ns, StiffRow& w) {
  w.beg = a < ns ? d.st_beg[a] : 0;
  w.len = a < ns ? (int)(d.st_end[a] - w.beg) : 0;
}

__device__ __forceinline__ void stiff_fetch(const Dev& d, StiffRow& w) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kPre; ++k) {
    const bool in = lane + 32 * k < w.len;
    w.v[k] = in ? __ldg(d.R_val + w.beg + lane + 32 * k) : 0.0;
    w.i[k] = in ? __ldg(d.R_idx + w.beg + lane + 32 * k) : -1;
  }
}

__device__ __forceinline__ double stiff_dot(const Dev& d, const StiffRow& w, const double* x) {
  const int lane = threadIdx.x & 31;
  double xv[kPre];
#pragma unroll
  for (int k = 0; k < kPre; ++k) xv[k] = w.i[k] >= 0 ? __ldcg(x + w.i[k]) : 0.0;
  double a[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const bool four = lane + 128 * h + 96 < w.len;
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (128 * h + 32 * k < w.len) {
        const double f = fma(w.v[4 * h + k], xv[4 * h + k], four ? a[k] : a[0]);
        if (four) a[k] = f;
        else if (w.i[4 * h + k] >= 0) a[0] = f;
      }
  }
  const double* val = d.R_val + w.beg;
  const int* idx = d.R_idx + w.beg;
  int e = lane + 256;
  for (; e + 96 < w.len; e += 128) {
#pragma unroll
    for (int k = 0; k < 4; ++k) a[k] = fma(__ldg(val + e + 32 * k), __ldcg(x + __ldg(idx + e + 32 * k)), a[k]);
  }
  for (; e < w.len; e += 32) a[0] = fma(__ldg(val + e), __ldcg(x + __ldg(idx + e)), a[0]);
  return warp_sum(w.len > 96 ? (a[0] + a[1]) + (a[2] + a[3]) : a[0]);
}

// E: unknowns per thread; LR: the preconditioner has the stiff rows' correction; MODE: an
// iteration of the FP64 (or refinement-pass) PCG, its start (r = rhs, dx = 0 given), or the two
// halves of an iteration of the PCG with residual replacement (before and after the FP64
// operator on dx; the second acts only when a replacement is due).
template <int E, bool LR, int MODE>
__global__ void __launch_bounds__(kTailThreads, 1) k_pcg_tail(Dev d, int npart, cudaGraphConditionalHandle h,
                                                             int set_cond) {
  __shared__ TailShared<E> s;
  Scal* sc = d.sc;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int nct = (int)gridDim.x, rank = (int)blockIdx.x;
  const bool lead = rank == 0 && tid == 0;
  const int done0 = sc->cg_done;
  if (MODE == TAIL_RU2 && !sc->ru_do) {
    if (lead && set_cond) cudaGraphSetConditional(h, done0 ? 0u : 1u);
    return;
  }
  if (done0 && MODE != TAIL_RU2) {
    if (lead && set_cond) cudaGraphSetConditional(h, 0u);
    return;
  }
  cl_arrive();
  // this CTA's unknowns: [j0, j1), whole blocks of 256; thread tid takes j0 + tid + 512 e
  const int nsys = (int)d.nsys, n = (int)d.n;
  const int per = ((nsys + nct - 1) / nct + 255) & ~255;
  const int j0 = rank * per, j1 = min(nsys, j0 + per);
  const int nw = min(kTailWarps, (max(j1 - j0, 0) + 31) >> 5);
  const bool act = w < nw;
  const int ns = LR ? sc->n_stiff : 0;
  // stiff rows: warp w of CTA c takes rows c + nct w, c + nct (w + 16), ...  What its first row
  // and this thread's columns need is fetched here where registers allow, else a phase ahead.
  constexpr bool kEarly = E <= 2;
  const int W = nct * kTailWarps, a0 = w * nct + rank;
  StiffRow row;
  int cb[E], cn[E], s0[E];             // the column's stiff entries: first and number; the first one's slot
  double v0[E], gv[kPre];              // and value; G^{-1}'s row
  auto fetch_cols = [&]() {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = j0 + tid + e * kTailThreads;
      const bool in = act && j < j1;
      const int2 run = in ? d.sc_run[j] : make_int2(0, 0);
      cb[e] = run.x;
      cn[e] = run.y;
    }
  };
  auto fetch_first = [&]() {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      v0[e] = cn[e] > 0 ? d.sc_val[cb[e]] : 0.0;
      s0[e] = cn[e] > 0 ? d.sc_slot[cb[e]] : 0;
    }
  };
  auto fetch_ginv = [&](int a) {
#pragma unroll
    for (int k = 0; k < kPre; ++k)
      gv[k] = (a < ns && lane + 32 * k < ns) ? d.Ginv[(int64_t)a * d.stiff_cap + lane + 32 * k] : 0.0;
  };
  if (LR && kEarly && ns > 0) {
    stiff_range(d, a0, ns, row);
    fetch_cols();
    fetch_ginv(a0);
  }
  double r[E], mi[E], p[E];
  if (MODE == TAIL_ITER || MODE == TAIL_RU) {
    double q[E], x[E];
    if (act) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int j = j0 + tid + e * kTailThreads;
        const bool in = j < j1;
        p[e] = in ? d.p[j] : 0.0;
        q[e] = in ? d.q[j] : 0.0;
        r[e] = in ? d.r[j] : 0.0;
        x[e] = in ? d.dx[j] : 0.0;
        mi[e] = in ? d.Minv[j] : 0.0;
      }
    }
    // p^T q: the column pass's block parts, in block order
    double pp = 0.0;
    if (tid < 256) {
      const double* part = d.partials + 16 * kMaxRedBlocks;
      double v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) v[k] = tid + 256 * k < npart ? part[tid + 256 * k] : 0.0;
      pp = v[0];
#pragma unroll
      for (int k = 1; k < 4; ++k)
        if (256 * k < npart) pp += v[k];
      for (int b = tid + 1024; b < npart; b += 256) pp += part[b];
    }
    if (LR && kEarly && ns > 0) {
      stiff_fetch(d, row);
      fetch_first();
    }
    const double pq = block_tree(pp, npart, s.w8);
    if (tid == 0) {
      const bool good = positive_finite(pq);            // else breakdown: keep the last iterate
      const double alpha = good ? sc->rz / pq : 0.0;
      s.alpha = alpha;
      s.stop = good ? 0 : 1;
      if (rank == 0) {
        sc->pq = pq;
        sc->alpha = alpha;
      }
    }
    __syncthreads();
    if (s.stop) {
      cl_wait();
      if (lead) {
        sc->cg_done = 1;
        if (!isfinite(sc->pq)) sc->status = DS_NUMERICAL;
        if (set_cond) cudaGraphSetConditional(h, 0u);
      }
      return;
    }
    if (act) {
      const double alpha = s.alpha;
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int j = j0 + tid + e * kTailThreads;
        x[e] = fma(alpha, p[e], x[e]);
        r[e] = fma(-alpha, q[e], r[e]);
        if (j < j1) {
          d.dx[j] = x[e];
          d.r[j] = r[e];
        }
      }
    }
  } else if (act) {
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = j0 + tid + e * kTailThreads;
      const bool in = j < j1;
      mi[e] = in ? d.Minv[j] : 0.0;
      if (MODE == TAIL_RU2) {
        p[e] = in ? d.p[j] : 0.0;
        r[e] = in ? d.rhs[j] - d.q[j] : 0.0;
        if (in) d.r[j] = r[e];
      } else {
        p[e] = 0.0;
        r[e] = in ? d.r[j] : 0.0;
      }
    }
  }
  double z[E];
  double rr = 0.0, rz = 0.0;
  if (act) {
#pragma unroll
    for (int e = 0; e < E; ++e) z[e] = r[e] * mi[e];
  }
  if (LR && ns > 0) {
    // z = z0 - M^{-1} A_s^T G^{-1} A_s z0, z0 = r / M
    if (act) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int j = j0 + tid + e * kTailThreads;
        if (j < j1) d.z[j] = z[e];
      }
    }
    if (!kEarly) stiff_range(d, a0, ns, row);
    cl_wait();
    cl_arrive();
    if (!kEarly || MODE == TAIL_INIT || MODE == TAIL_RU2) stiff_fetch(d, row);
    if (!kEarly) fetch_cols();
    else if (MODE == TAIL_INIT || MODE == TAIL_RU2) fetch_first();
    cl_wait();
    for (int a = a0; a < ns; a += W) {
      if (a != a0) {
        stiff_range(d, a, ns, row);
        stiff_fetch(d, row);
      }
      const double u = stiff_dot(d, row, d.z);
      if (lane < nct) cl_store(&s.u[a], lane, u);
    }
    if (!kEarly) fetch_ginv(a0);
    __syncwarp();
    cl_arrive();
    if (!kEarly) fetch_first();
    cl_wait();
    // t = G^{-1} u, one warp per row
    for (int a = a0; a < ns; a += W) {
      const double* gr = d.Ginv + (int64_t)a * d.stiff_cap;
      if (a != a0) fetch_ginv(a);
      double t = 0.0;
#pragma unroll
      for (int k = 0; k < kPre; ++k)
        if (32 * k < ns) t = fma(gv[k], lane + 32 * k < ns ? s.u[lane + 32 * k] : 0.0, t);
      for (int b = 32 * kPre + lane; b < ns; b += 32) t = fma(gr[b], s.u[b], t);
      t = warp_sum(t);
      if (lane < nct) cl_store(&s.t[a], lane, t);
    }
    __syncwarp();
    cl_arrive();
    cl_wait();
    if (act) {
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (cn[e] > 0) {
          double acc = v0[e] * s.t[s0[e]];
          for (int t = 1; t < cn[e]; ++t) acc = fma(d.sc_val[cb[e] + t], s.t[d.sc_slot[cb[e] + t]], acc);
          z[e] -= mi[e] * acc;
        }
    }
  }
  // r^T z and ||r||^2 over the cluster; warp 0 decides and forms beta
  if (LR) __syncthreads();             // s.t is read, its memory becomes s.red
  const int nvb = (max(j1 - j0, 0) + 255) >> 8, nvw = 8 * nvb;   // blocks and warps of this CTA's values
  if (act) {
#pragma unroll
    for (int e = 0; e < E; ++e) rr = fma(r[e], r[e], rr);
  }
  s.rr[w * 33 + lane] = rr;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int j = j0 + tid + e * kTailThreads;
    if (w + 16 * e < nvw) s.red[(w + 16 * e) * 33 + lane] = j < j1 ? r[e] * z[e] : 0.0;
  }
  __syncthreads();
  if (E > 4) {
    if (tid < nvw) s.wsum[tid] = tree32(s.red + tid * 33);
    if (w >= 4) tree_runs(s.rr, nw, s.rw, 4);
  } else {
    tree_runs(s.red, nvw, s.wsum, 0);
    if (w >= 12) tree_runs(s.rr, nw, s.rw, 12);
  }
  __syncthreads();
  if (!(LR && ns > 0)) cl_wait();
  const int b0 = j0 >> 8, nb = (nsys + 255) >> 8;
  if (w * 4 < nvb) {
    // block b of this CTA by 8 lanes: its tree over the 8 warps, to every CTA
    const int b = tid >> 3, g = tid & 7;
    double t = b < nvb ? s.wsum[8 * b + g] : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (b < nvb)
      for (int c = g; c < nct; c += 8) cl_store(&s.part[b0 + b], c, t);
  }
  if (w == kTailWarps - 1) {
    rr = lane < nw ? s.rw[lane] : 0.0;
#pragma unroll
    for (int o = kTailWarps / 2; o > 0; o >>= 1) rr += __shfl_xor_sync(0xffffffffu, rr, o);
    if (lane < nct) cl_store(&s.xrr[rank], lane, rr);
  }
  __syncwarp();
  // the scalars, read before the barrier after which CTA 0 writes them: thread 0 forms beta,
  // the first thread of warp 1 decides
  double rz_old = 0.0, tol2 = 0.0, due2 = 0.0, outer = 0.0;
  int it = 0, mx = 0;
  if (lane == 0 && w < 2) {
    rz_old = sc->rz;
    tol2 = MODE == TAIL_ITER ? sc->tol2 : sc->tol2_outer;
    outer = sc->rr_outer;
    it = sc->cg_iter;
    mx = sc->cg_max;
    if (MODE == TAIL_RU) due2 = sc->refine_eta * sc->refine_eta * sc->rr_ref;
  }
  cl_arrive();
  cl_wait();
  rz = block_tree(tid < nb ? s.part[tid] : 0.0, nb, s.w8);      // nb <= kTailBlocks
  if (w < 2) {
    rr = lane < nct ? s.xrr[lane] : 0.0;
    if (w == 1 || MODE == TAIL_RU2) {
#pragma unroll
      for (int o = kTailCtas / 2; o > 0; o >>= 1) rr += __shfl_xor_sync(0xffffffffu, rr, o);
    }
    // no progress since the last replacement (the true residual fell by less than a tenth: the
    // kept direction has lost conjugacy to the coarse operator's drift): restart the Krylov
    // process from this residual
    if (tid == 0) {
      const double beta = MODE == TAIL_INIT || (MODE == TAIL_RU2 && rr > 0.81 * outer) ? 0.0 : rz / rz_old;
      s.beta = beta;
      s.rz = rz;
    }
    if (tid == 32) {
      bool stop = false;
      if (MODE != TAIL_INIT) {
        if (MODE != TAIL_RU2) it += 1;
        const bool fin = isfinite(rr), conv = fin && rr <= tol2;
        const bool due = MODE == TAIL_RU && fin && (conv || rr <= due2 || it >= mx);
        stop = MODE == TAIL_RU ? !fin || due : done0 || !fin || conv || it >= mx;
        if (rank == 0) {
          sc->cg_iter = it;
          sc->rr = rr;
          if (!fin) sc->status = DS_NUMERICAL;
          if (MODE == TAIL_RU) {
            sc->ru_do = due ? 1 : 0;
            if (!fin) sc->cg_done = 1;
          } else {
            if (stop) sc->cg_done = 1;
            if (conv) sc->cg_conv = 1;
            if (set_cond) cudaGraphSetConditional(h, stop ? 0u : 1u);
          }
          if (MODE == TAIL_RU2) {
            sc->refine_it += 1;
            sc->rr_ref = rr;
            sc->rr_outer = rr;
            if (conv) sc->cg_conv_outer = 1;
          }
        }
      } else if (rank == 0 && set_cond) {
        cudaGraphSetConditional(h, 1u);
      }
      s.stop = stop ? 1 : 0;
    }
  }
  __syncthreads();
  if (s.stop) return;
  if (lead) {
    sc->rz = s.rz;
    if (MODE != TAIL_INIT) sc->beta = s.beta;
  }
  if (act) {
    const double beta = s.beta;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int j = j0 + tid + e * kTailThreads;
      if (MODE != TAIL_INIT) z[e] = fma(beta, p[e], z[e]);
      if (j < j1) d.p[j] = z[e];
    }
    if (d.p32) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int j = j0 + tid + e * kTailThreads;
        if (j < j1) d.p32[j] = (float)z[e];
      }
    }
    if (d.p_df) {
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int j = j0 + tid + e * kTailThreads;
        if (j < min(j1, n)) d.p_df[j] = df_split(z[e]);
      }
    }
  }
  if (LR && ns > 0 && d.p32) {
    // reduced storage: u_a = theta_a (A_a . p), the stiff rows' exact part of the next K~ p
    if (!kEarly || ns > W) {
      stiff_range(d, a0, ns, row);
      stiff_fetch(d, row);
    }
    cl_arrive();
    cl_wait();
    for (int a = a0; a < ns; a += W) {
      if (a != a0) {
        stiff_range(d, a, ns, row);
        stiff_fetch(d, row);
      }
      const double u = stiff_dot(d, row, d.p);
      if (lane == 0) d.us2[a] = d.theta[d.stiff_k[a]] * u;
    }
  }
}

// A cluster of `ctas` CTAs; the attribute lives as long as the configuration is used.
cudaLaunchConfig_t tail_config(int ctas, cudaStream_t st, cudaLaunchAttribute* at) {
  cudaLaunchConfig_t c{};
  c.gridDim = dim3((unsigned)ctas);
  c.blockDim = dim3(kTailThreads);
  c.stream = st;
  at->id = cudaLaunchAttributeClusterDimension;
  at->val.clusterDim.x = (unsigned)ctas;
  at->val.clusterDim.y = 1;
  at->val.clusterDim.z = 1;
  c.attrs = at;
  c.numAttrs = 1;
  return c;
}

template <int E, bool LR, int MODE>
cudaError_t launch_one(const Dev& d, int ctas, int npart, cudaGraphConditionalHandle h, int set_cond, cudaStream_t st) {
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t c = tail_config(ctas, st, &at);
  return cudaLaunchKernelEx(&c, k_pcg_tail<E, LR, MODE>, d, npart, h, set_cond);
}

// Sets a form's attributes on the current device and asks whether a cluster of it finds room there.
template <int E, bool LR, int MODE>
bool places_one(int ctas) {
  auto* f = k_pcg_tail<E, LR, MODE>;
  cudaLaunchAttribute at;
  const cudaLaunchConfig_t c = tail_config(ctas, 0, &at);
  int clusters = 0;
  const bool ok = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
                  // one CTA an SM: no more shared memory taken from the L1 than it needs (see k_gram_G's)
                  cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxL1) == cudaSuccess &&
                  cudaOccupancyMaxActiveClusters(&clusters, f, &c) == cudaSuccess;
  if (!ok) cudaGetLastError();
  return ok && clusters > 0;
}

template <int E, bool LR>
cudaError_t launch_mode(const Dev& d, int mode, int ctas, int npart, cudaGraphConditionalHandle h, int set_cond,
                        cudaStream_t st) {
  switch (mode) {
    case TAIL_INIT: return launch_one<E, LR, TAIL_INIT>(d, ctas, npart, h, set_cond, st);
    case TAIL_RU: return launch_one<E, LR, TAIL_RU>(d, ctas, npart, h, set_cond, st);
    case TAIL_RU2: return launch_one<E, LR, TAIL_RU2>(d, ctas, npart, h, set_cond, st);
    default: return launch_one<E, LR, TAIL_ITER>(d, ctas, npart, h, set_cond, st);
  }
}

// CTAs of the cluster: a small problem's barriers are cheaper among fewer CTAs, and a small
// cluster finds room beside other solves sooner (with 512 unknowns each of 8 CTAs still has a
// thread for every one of its own).
int tail_ctas(int64_t nsys) { return nsys <= kTailSmall ? 8 : 16; }

// f(integral_constant E, bool_constant LR, CTAs) for the form that covers a system.
template <typename F>
auto tail_form(const Dev& d, int precond, F f) {
  const int ctas = tail_ctas(d.nsys);
  const int64_t cta_n = ((d.nsys + ctas - 1) / ctas + 255) & ~(int64_t)255;
  const int64_t per = (cta_n + kTailThreads - 1) / kTailThreads;
  const bool lr = precond == PC_JACOBI_LR && d.m > 0;
  auto go = [&](auto ec) { return lr ? f(ec, std::true_type{}, ctas) : f(ec, std::false_type{}, ctas); };
  if (per <= 1) return go(std::integral_constant<int, 1>{});
  if (per <= 2) return go(std::integral_constant<int, 2>{});
  if (per <= 4) return go(std::integral_constant<int, 4>{});
  return go(std::integral_constant<int, kTailMaxE>{});
}

cudaError_t launch_tail(const Dev& d, int precond, int mode, int npart, cudaGraphConditionalHandle h, bool set_cond,
                        cudaStream_t st) {
  return tail_form(d, precond, [&](auto ec, auto lr, int ctas) {
    return launch_mode<decltype(ec)::value, decltype(lr)::value>(d, mode, ctas, npart, h, set_cond ? 1 : 0, st);
  });
}

// The cluster form covers a system of this size and preconditioner.
bool tail_covers(const Dev& d, int precond) {
  if (precond != PC_JACOBI && precond != PC_JACOBI_LR) return false;
  const bool lr = precond == PC_JACOBI_LR && d.m > 0;
  return d.nsys <= (lr || d.storage != ST_F64 ? kTailMaxN : kTailPlainN);
}

}  // namespace

bool tail_runs(const Dev& d, int precond) { return d.cluster && !(d.crowd && !d.aug) && tail_covers(d, precond); }

// 16 SMs of one processing cluster are not a given: a process may be confined to fewer, and then every
// launch would fail where the whole-chip kernels run.
bool tail_places(const Dev& d, int precond) {
  if (!tail_covers(d, precond)) return false;
  return tail_form(d, precond, [&](auto ec, auto lr, int ctas) {
    constexpr int E = decltype(ec)::value;
    constexpr bool LR = decltype(lr)::value;
    return places_one<E, LR, TAIL_ITER>(ctas) && places_one<E, LR, TAIL_INIT>(ctas) &&
           (d.storage == ST_F64 || (places_one<E, LR, TAIL_RU>(ctas) && places_one<E, LR, TAIL_RU2>(ctas)));
  });
}

cudaError_t launch_tail_init(const Dev& d, int precond, cudaGraphConditionalHandle h, cudaStream_t st) {
  return launch_tail(d, precond, TAIL_INIT, 0, h, h != 0, st);
}
cudaError_t launch_tail_iter(const Dev& d, int precond, int npart, cudaGraphConditionalHandle h, bool in_graph,
                             cudaStream_t st) {
  return launch_tail(d, precond, TAIL_ITER, npart, h, in_graph, st);
}
cudaError_t launch_tail_ru(const Dev& d, int precond, int npart, cudaStream_t st) {
  return launch_tail(d, precond, TAIL_RU, npart, 0, false, st);
}
cudaError_t launch_tail_ru2(const Dev& d, int precond, cudaGraphConditionalHandle h, bool in_graph, cudaStream_t st) {
  return launch_tail(d, precond, TAIL_RU2, 0, h, in_graph, st);
}

}  // namespace ipmk
