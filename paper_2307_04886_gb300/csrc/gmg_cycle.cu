// V-cycle of Alg. 2 on the GPU and the outer iterations of Alg. 1.
//
// Layout: every level is renumbered colour by colour; the off-diagonal part
// of A_l is a sliced ELL with 32-row slices stored [k][lane], so the 32 lanes
// of a warp read 32 consecutive values and column indices per k.  A
// Gauss-Seidel colour is one launch over that colour's slices: rows of a
// colour are never adjacent, so every row reads only other colours' entries of
// x and the in-place update equals sequential Gauss-Seidel in colour order.
// Levels with long rows split each row over G warps (G = 1, 2, 4 or 8; warp
// `part` takes k = part, part + G, ...), combining the G partial sums in a
// fixed order, so the dependent-load chain per row is G times shorter.
// The restriction P_l^T is a sliced ELL over the coarse rows (a gather: no
// atomics, a fixed summation order); it also clears the coarse iterate (the
// recursive call of Alg. 2 starts from zero).  The prolongation reads three
// packed (index, weight) slots per fine row.  The coarsest level applies the
// explicit FP64 inverse of its operator as a warp-per-row GEMV (the cluster
// launch, gmg_cluster.cu, has its own coarsest solve).
//
// Launches use programmatic dependent launch: a kernel may start while its
// predecessor drains; it loads only setup-time data (matrix values, column
// indices, inverse diagonal) before `griddepcontrol.wait`, and everything the
// previous kernel may write after it.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <string>
#include <type_traits>
#include <utility>

#include "gmg_cycle.cuh"

namespace gmg {


// ------------------------------------------------------------------ kernels

constexpr int kPrefetch = 8;  // matrix entries per lane loaded before the dependency wait

// Per-lane view of a sliced-ELL row split over G warps.
struct RowPart {
  bool active;
  int nk;        // entries of this row handled by this warp
  int64_t e;     // first entry
  int64_t row;
};

template <int G>
__device__ __forceinline__ RowPart row_part(int64_t s, int64_t s_end, const int64_t* __restrict__ ptr,
                                            const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                            int part, int lane) {
  RowPart p{false, 0, 0, 0};
  if (s < s_end) {
    p.active = lane < nrow[s];
    const int64_t e0 = ptr[s];
    const int w = (int)((ptr[s + 1] - e0) >> 5);
    p.nk = (p.active && part < w) ? (w - part + G - 1) / G : 0;
    p.e = e0 + (int64_t)part * 32 + lane;
    p.row = row0[s] + lane;
  }
  return p;
}

// sum_k a_rk x_{c_rk} over this warp's share of row r; the first kPrefetch
// values and columns were loaded before the wait.
template <class T, int G>
__device__ __forceinline__ T row_dot(const RowPart& p, const T (&pv)[kPrefetch], const int (&pc)[kPrefetch],
                                     const int32_t* __restrict__ col, const T* __restrict__ val, const T* x) {
  T acc = 0;
#pragma unroll
  for (int q = 0; q < kPrefetch; ++q)
    if (q < p.nk) acc += pv[q] * x[pc[q]];
  for (int q = kPrefetch; q < p.nk; ++q) {
    const int64_t e = p.e + (int64_t)q * G * 32;
    acc += val[e] * x[col[e]];
  }
  return acc;
}

template <class T, int G>
__device__ __forceinline__ void prefetch_row(const RowPart& p, const int32_t* __restrict__ col,
                                             const T* __restrict__ val, T (&pv)[kPrefetch], int (&pc)[kPrefetch]) {
#pragma unroll
  for (int q = 0; q < kPrefetch; ++q) {
    if (q < p.nk) {
      const int64_t e = p.e + (int64_t)q * G * 32;
      pv[q] = val[e];
      pc[q] = col[e];
    } else {
      pv[q] = 0;
      pc[q] = 0;
    }
  }
}

// Combines the G partial sums of a row in warp order (part 0 first).
template <class T, int G>
__device__ __forceinline__ T combine_parts(T acc, int warp, int lane) {
  if constexpr (G > 1) {
    __shared__ T red[8][32];
    red[warp][lane] = acc;
    __syncthreads();
    if (warp % G == 0) {
#pragma unroll
      for (int g = 1; g < G; ++g) acc += red[warp + g][lane];
    }
  }
  return acc;
}

// Sums of NS values per thread over a block of 256 threads in a fixed order
// (the tree t += t + o, o = 128 .. 1); thread 0 gets them.  The last five
// levels are one warp's shuffles: a level is then one dependent FP64 addition,
// without the barrier and the shared-memory round trip.
template <int NS>
__device__ __forceinline__ void block_sums(double (&v)[NS], double (*red)[256]) {
  const int t = threadIdx.x;
#pragma unroll
  for (int k = 0; k < NS; ++k) red[k][t] = v[k];
  __syncthreads();
#pragma unroll
  for (int o = 128; o >= 32; o >>= 1) {
    if (t < o) {
#pragma unroll
      for (int k = 0; k < NS; ++k) {
        v[k] += red[k][t + o];
        red[k][t] = v[k];
      }
    }
    if (o > 32) __syncthreads();
  }
  if (t < 32) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int k = 0; k < NS; ++k) v[k] += __shfl_down_sync(0xffffffffu, v[k], o);
  }
}

// Sums of partial[k * stride + (0 .. count)), k < NS, by one block of 256
// threads in a fixed order (strided per-thread sums, then the tree); thread 0
// gets them.  Partials written by other blocks of the same grid are read
// through L2, four at a time.
template <int NS>
__device__ __forceinline__ void block_final_sums(int count, const double* partial, int stride, double (&v)[NS],
                                                 double (*red)[256]) {
#pragma unroll
  for (int k = 0; k < NS; ++k) v[k] = 0.0;
  for (int i0 = threadIdx.x; i0 < count; i0 += 1024) {
    double p[NS][4];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < NS; ++k) p[k][q] = i0 + 256 * q < count ? __ldcg(partial + k * stride + i0 + 256 * q) : 0.0;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < NS; ++k) v[k] += p[k][q];
  }
  __syncthreads();
  block_sums<NS>(v, red);
}

// True in the one block of the grid that arrives last (after every block has
// written its partial sums); that block then finishes the reduction, so no
// separate single-block kernel is launched.  `counter` returns to 0.
__device__ bool last_block(int* counter) {
  __shared__ int is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    is_last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
    if (is_last) *counter = 0;
  }
  __syncthreads();
  if (is_last) __threadfence();
  return is_last != 0;
}

// One colour of a Gauss-Seidel sweep: x_r = (b_r - sum_{k != r} a_rk x_k) / a_rr
// for the rows of slices [s0, s1).  The FP32 one-warp-per-slice form (the
// finest level) is held to 32 registers so that 8 CTAs fit per SM and a whole
// colour of the finest level is resident in one wave (measured: 5.9 -> 5.6 us
// per colour on the 1M-vertex torus).
template <class T, int G>
__global__ void __launch_bounds__(256, (G == 1 && sizeof(T) == 4) ? 8 : 1) k_gs(int64_t s0, int64_t s1, const int64_t* __restrict__ ptr,
                                            const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                            const int32_t* __restrict__ col, const T* __restrict__ val,
                                            const T* __restrict__ dinv, const T* b, T* x) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % G;
  const int64_t s = s0 + (int64_t)blockIdx.x * (8 / G) + warp / G;
  const RowPart p = row_part<G>(s, s1, ptr, row0, nrow, part, lane);
  T pv[kPrefetch];
  int pc[kPrefetch];
  prefetch_row<T, G>(p, col, val, pv, pc);
  const T di = (part == 0 && p.active) ? dinv[p.row] : T(0);
  pdl_wait();
  pdl_trigger();
  // b is issued with the gathers: after the barrier of combine_parts its load
  // would be one more dependent round trip to L2
  const T bv = (part == 0 && p.active) ? b[p.row] : T(0);
  T acc = row_dot<T, G>(p, pv, pc, col, val, x);
  acc = combine_parts<T, G>(acc, warp, lane);
  if (part == 0 && p.active) x[p.row] = (bv - acc) * di;
}

// The start of a device-driven solve (one thread): the initial relative
// residual, and whether the right-hand side is nonzero and both are finite
// (the iterations of a solve that must not run are discarded by k_store).
__device__ void start_check(double* sc, double* hist) {
  const double nb = sqrt(sc[S_NB2]), rel = sqrt(sc[S_RR]) / nb;
  hist[0] = rel;
  sc[S_OK] = isfinite(nb) && nb > 0.0 && isfinite(rel) ? 1.0 : 0.0;
}

// The convergence test of the device-side loop (one thread): advances the
// iteration counter it[0], records rel = ||r|| / ||b|| (same arithmetic as the
// host test) and keeps the loop going while rel is finite, above the
// tolerance and the counter below it[1].
__device__ void iter_check(const double* sc, int* it, double* hist, cudaGraphConditionalHandle h) {
  const int k = ++it[0];
  const double rel = sqrt(sc[S_RR]) / sqrt(sc[S_NB2]);
  hist[k] = rel;
  const bool go = isfinite(rel) && !(rel <= sc[S_TOL]) && k < it[1];
  cudaGraphSetConditional(h, go ? 1u : 0u);
}

// What the last block of a residual with a norm does with ||r||^2 besides
// storing it: nothing, the test of a solve's start (start_check), or the
// convergence test of the device-side loop (iter_check).
enum { kNormOnly = 0, kNormStart = 1, kNormIter = 2 };
struct NormEnd {
  double* partial;  // one sum of r^2 per block
  int* counter;
  double* sc;
  int* it;
  double* hist;
  cudaGraphConditionalHandle h;
  int what;
};

// r = b - A x over all slices.  With NORM also ||r||^2 into sc[S_RR]: fixed
// block sums, added in block order by the last block, which then runs the
// test named in `end` (a separate one-block sum and a one-thread test cost a
// launch each: 5 us per iteration of the refinement modes).  With NORM a block
// takes every gridDim-th group of slices: a block's reduction (nine dependent
// FP64 additions, a fence and an atomic, about 3 us) then falls due once per
// resident block and not once per 256 rows (1M-vertex torus: 59 -> 32 us).
template <class T, int G, bool NORM>
__global__ void __launch_bounds__(256, NORM ? 4 : 1) k_residual(int64_t nslice, const int64_t* __restrict__ ptr,
                                                  const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                                  const int32_t* __restrict__ col, const T* __restrict__ val,
                                                  const T* __restrict__ diag, const T* x, const T* b, T* r,
                                                  NormEnd end) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % G;
  double sq = 0.0;
  bool first = true;
  for (int64_t s0 = (int64_t)blockIdx.x * (8 / G); s0 < nslice; s0 += (int64_t)gridDim.x * (8 / G)) {
    const RowPart p = row_part<G>(s0 + warp / G, nslice, ptr, row0, nrow, part, lane);
    T pv[kPrefetch];
    int pc[kPrefetch];
    prefetch_row<T, G>(p, col, val, pv, pc);
    const T d = (part == 0 && p.active) ? diag[p.row] : T(0);
    if (first) {
      pdl_wait();
      pdl_trigger();
      first = false;
    } else if constexpr (G > 1) {
      __syncthreads();  // the sums of the group before have been read
    }
    const bool own = part == 0 && p.active;
    const T bv = own ? b[p.row] : T(0), xv = own ? x[p.row] : T(0);  // issued with the gathers
    T acc = row_dot<T, G>(p, pv, pc, col, val, x);
    acc = combine_parts<T, G>(acc, warp, lane);
    if (own) {
      const T rv = bv - (acc + d * xv);
      r[p.row] = rv;
      if constexpr (NORM) sq += to_f64(rv) * to_f64(rv);
    }
    if constexpr (!NORM) break;
  }
  if constexpr (NORM) {
    __shared__ double red[1][256];
    double v[1] = {sq};
    block_sums<1>(v, red);
    if (threadIdx.x == 0) end.partial[blockIdx.x] = v[0];
    if (last_block(end.counter)) {
      block_final_sums<1>(gridDim.x, end.partial, 0, v, red);
      if (threadIdx.x == 0) {
        end.sc[S_RR] = v[0];
        if (end.what == kNormStart) start_check(end.sc, end.hist);
        if (end.what == kNormIter) iter_check(end.sc, end.it, end.hist, end.h);
      }
    }
  }
}

// q = A p (FP64) and p.q into *out; blocks take every gridDim-th group of
// eight slices, as in k_residual.  What bounds it then is the FP64 pipe (a
// warp's FP64 instruction takes 64 cycles of its sub-partition): eight per
// slice of a mesh Laplacian are 14 us on the 1M-vertex torus.  47 -> 27 us.
__global__ void __launch_bounds__(256, 4) k_spmv_dot(int64_t nslice, const int64_t* __restrict__ ptr,
                                                  const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                                  const int32_t* __restrict__ col, const double* __restrict__ val,
                                                  const double* __restrict__ diag, const double* p,
                                                  double* q, double* __restrict__ partial, int* counter,
                                                  double* out) {
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * 8;
  double pq = 0.0;
  bool first = true;
  for (int64_t s = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5); s < nslice || first; s += step) {
    const RowPart rp = row_part<1>(s, nslice, ptr, row0, nrow, 0, lane);
    double pv[kPrefetch];
    int pc[kPrefetch];
    prefetch_row<double, 1>(rp, col, val, pv, pc);
    const double d = rp.active ? diag[rp.row] : 0.0;
    if (first) {
      pdl_wait();
      pdl_trigger();
      first = false;
    }
    if (rp.active) {
      const double pr = p[rp.row];
      const double acc = row_dot<double, 1>(rp, pv, pc, col, val, p) + d * pr;
      q[rp.row] = acc;
      pq += pr * acc;
    }
  }
  __shared__ double red[1][256];
  double v[1] = {pq};
  block_sums<1>(v, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = v[0];
  if (last_block(counter)) {
    block_final_sums<1>(gridDim.x, partial, 0, v, red);
    if (threadIdx.x == 0) *out = v[0];
  }
}

// bc = P^T r (gather over the transpose) and xc = 0 (the coarse iterate of the
// recursive call starts from zero).
template <class T>
__global__ void __launch_bounds__(256) k_restrict(int64_t nslice, const int64_t* __restrict__ ptr,
                                                  const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                                  const int32_t* __restrict__ col, const T* __restrict__ w,
                                                  const T* r, T* bc, T* xc, const T* __restrict__ dinvc,
                                                  int64_t nc0) {
  const int lane = threadIdx.x & 31;
  const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const RowPart p = row_part<1>(s, nslice, ptr, row0, nrow, 0, lane);
  T pv[kPrefetch];
  int pc[kPrefetch];
  prefetch_row<T, 1>(p, col, w, pv, pc);
  const bool c0 = p.active && p.row < nc0;
  const T dc = c0 ? dinvc[p.row] : T(0);
  pdl_wait();
  pdl_trigger();
  if (!p.active) return;
  const T acc = row_dot<T, 1>(p, pv, pc, col, w, r);
  bc[p.row] = acc;
  // the first Gauss-Seidel colour of the coarse pre-smoothing from x = 0:
  // (b - 0) / a_ii for the rows of colour 0 (the first nc0 rows)
  xc[p.row] = c0 ? (acc - T(0)) * dc : T(0);
}

// x += P u (three packed slots per fine row).
template <class T>
__global__ void __launch_bounds__(256) k_prolong(int64_t n, const int32_t* __restrict__ idx, const T* __restrict__ w,
                                                 const T* u, T* x) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int i0 = 0, i1 = 0, i2 = 0;
  T w0 = 0, w1 = 0, w2 = 0;
  if (i < n) {
    i0 = idx[3 * i];
    i1 = idx[3 * i + 1];
    i2 = idx[3 * i + 2];
    w0 = w[3 * i];
    w1 = w[3 * i + 1];
    w2 = w[3 * i + 2];
  }
  pdl_wait();
  pdl_trigger();
  if (i < n) x[i] += w0 * u[i0] + w1 * u[i1] + w2 * u[i2];
}

// x = Ainv b, one warp per row, FP64 accumulation in both precisions.
template <class T>
__global__ void __launch_bounds__(256) k_coarse(int n, const double* __restrict__ Ainv, const T* b, T* x) {
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  pdl_wait();
  pdl_trigger();
  if (row >= n) return;
  const double* a = Ainv + (int64_t)row * n;
  double s = 0.0;
  for (int j = lane; j < n; j += 32) s += a[j] * to_f64(b[j]);
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) x[row] = (T)s;
}

#define GRID_LOOP(i, n) \
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (n); i += (int64_t)gridDim.x * blockDim.x)

__global__ void k_gather(int64_t n, const int32_t* __restrict__ perm, const double* src, double* dst) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) dst[i] = src[perm[i]];
}
// The end of a single V-cycle: dst[perm] = src, or NaN everywhere if a bounded
// wait of its cluster launch gave up (the call does not synchronise, so that it
// cannot return the status).
__global__ void k_scatter_cycle(int64_t n, const int32_t* __restrict__ perm, const double* src, double* dst,
                                const int* wait_failed) {
  pdl_wait();
  pdl_trigger();
  const bool failed = *wait_failed != 0;
  GRID_LOOP(i, n) dst[perm[i]] = failed ? __longlong_as_double(0x7FF8000000000000LL) : src[i];
}
__global__ void k_scatter_vec(int64_t n, const int32_t* __restrict__ perm, const double* src, double* dst) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) dst[perm[i]] = src[i];
}
__global__ void k_d2f(int64_t n, const double* a, float* b) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) b[i] = f32_rn(a[i]);
}
// b32 = (float) r and x32 = 0: the right-hand side and zero initial guess of
// a correction cycle MGI(0, r); the rows of colour 0 (the first n0) take
// their first Gauss-Seidel update from x = 0 right away, (b - 0) / a_ii.
__global__ void k_d2f_zero(int64_t n, const double* r, float* b32, float* x32, const float* __restrict__ dinv32,
                           int64_t n0) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) {
    const float bi = f32_rn(r[i]);
    b32[i] = bi;
    x32[i] = i < n0 ? (bi - 0.f) * dinv32[i] : 0.f;
  }
}
__global__ void k_f2d(int64_t n, const float* a, double* b) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) b[i] = f64_of(a[i]);
}
// x += (double) e
__global__ void k_add_f2d(int64_t n, const float* e, double* x) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) x[i] += f64_of(e[i]);
}

// The vectors of a solve in the level's numbering, bs = b[perm] and
// xs = x[perm], ||b||^2 into sc[S_NB2], and the solve's tolerance, iteration
// counter and limit: one launch instead of two gathers, two reduction kernels
// and two copies from the host; the bounded waits' error word is cleared.  Sums: fixed grid (kRedBlocks x 256), fixed
// per-thread ranges, fixed tree.
__global__ void __launch_bounds__(256, 4) k_load(int64_t n, const int32_t* __restrict__ perm,
                                              const double* __restrict__ b, const double* __restrict__ x,
                                              double* __restrict__ bs, double* __restrict__ xs,
                                              double* __restrict__ partial, int* counter, double* sc, int* it,
                                              double tol, int max_iter, int* wait_failed) {
  __shared__ double red[1][256];
  pdl_wait();
  pdl_trigger();
  double s = 0.0;
#pragma unroll 2
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const int32_t o = perm[i];
    const double bi = b[o];
    bs[i] = bi;
    xs[i] = x[o];
    s += bi * bi;
  }
  double v[1] = {s};
  block_sums<1>(v, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = v[0];
  if (last_block(counter)) {
    block_final_sums<1>(gridDim.x, partial, 0, v, red);
    if (threadIdx.x == 0) {
      sc[S_NB2] = v[0];
      sc[S_TOL] = tol;
      it[0] = 0;
      it[1] = max_iter;
      *wait_failed = 0;  // what an earlier call on the handle left there is not this solve's
    }
  }
}

// The end of a device-driven solve: x[perm] = xs unless the start's test
// failed, and the solve's report straight into pinned host memory (block 0):
// the host reads it after the one synchronisation of the solve.
__global__ void __launch_bounds__(256) k_store(int64_t n, const int32_t* __restrict__ perm,
                                               const double* __restrict__ xs, double* __restrict__ x,
                                               const double* sc, const int* it, const double* hist,
                                               const int* status, double* rep) {
  pdl_wait();
  pdl_trigger();
  if (blockIdx.x == 0) {
    const int k = it[0];
    if (threadIdx.x == 0) {
      rep[REP_NB2] = sc[S_NB2];
      rep[REP_RR] = sc[S_RR];
      rep[REP_OK] = sc[S_OK];
      rep[REP_ITERS] = k;
      rep[REP_REL] = hist[k];
      rep[REP_PIVOT] = status[1];
      rep[REP_WAIT] = status[3];
    }
    for (int i = threadIdx.x; i <= k && i < REP_HIST_CAP; i += 256) rep[REP_HIST + i] = hist[i];
  }
  if (sc[S_OK] != 1.0) return;
  GRID_LOOP(i, n) x[perm[i]] = xs[i];
}

// PCG scalars live on the device (slots S_*): r.z, p.Ap, the Polak-Ribiere
// numerator z.(r - r_old), beta.
//
// alpha = rz / pq; r_old = r; x += alpha p; r -= alpha q; rr = r.r into
// sc[S_RR] (partials, finished by the last block); and the initial iterate of
// the next preconditioning cycle MGI(0, r): with an FP32 cycle its right-hand
// side b32 = (float) r and x32 (as k_d2f_zero), with an FP64 cycle (which
// reads r itself as its right-hand side) z64.  The rows of colour 0 (the
// first n0) take their first Gauss-Seidel update from zero, (r - 0) / a_ii.
// With `check` the last block also runs the convergence test of the
// device-side loop.  Grid: kRedBlocks x 256.
template <class Z>
__global__ void __launch_bounds__(256, 4) k_pcg_axpy(int64_t n, double* sc, const double* __restrict__ p,
                                                  const double* __restrict__ q, double* __restrict__ x,
                                                  double* __restrict__ r, double* __restrict__ rold,
                                                  float* __restrict__ b32, Z* __restrict__ z0,
                                                  const Z* __restrict__ dinv, int64_t n0,
                                                  double* __restrict__ partial, int* counter, int check, int* it,
                                                  double* hist, cudaGraphConditionalHandle h) {
  __shared__ double red[1][256];
  pdl_wait();
  pdl_trigger();
  const double alpha = sc[S_RZ] / sc[S_PQ];
  double rr = 0.0;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const double ri = r[i];
    rold[i] = ri;
    x[i] += alpha * p[i];
    const double rn = ri - alpha * q[i];
    r[i] = rn;
    if constexpr (sizeof(Z) == 4) {
      const float bi = f32_rn(rn);
      b32[i] = bi;
      z0[i] = i < n0 ? (bi - 0.f) * dinv[i] : 0.f;
    } else {
      z0[i] = i < n0 ? (rn - 0.0) * dinv[i] : 0.0;
    }
    rr += rn * rn;
  }
  double v[1] = {rr};
  block_sums<1>(v, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = v[0];
  if (last_block(counter)) {
    block_final_sums<1>(gridDim.x, partial, 0, v, red);
    if (threadIdx.x == 0) {
      sc[S_RR] = v[0];
      if (check) iter_check(sc, it, hist, h);
    }
  }
}

// z = the preconditioned residual (the cycle's output, FP32 or FP64); the
// Polak-Ribiere numerator z.(r - r_old) and r.z, partial sums finished by the
// last block, which sets beta = num / rz_old and rz = r.z for the next
// iteration.  Grid: kRedBlocks x 256.
template <class Z>
__global__ void __launch_bounds__(256, 4) k_pcg_zdots(int64_t n, const Z* __restrict__ z, const double* __restrict__ r,
                                                   const double* __restrict__ rold, double* __restrict__ partial,
                                                   int* counter, double* sc) {
  __shared__ double red[2][256];
  pdl_wait();
  pdl_trigger();
  double num = 0.0, rz = 0.0;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const double zi = to_f64(z[i]), ri = r[i];
    num += zi * (ri - rold[i]);
    rz += ri * zi;
  }
  double v[2] = {num, rz};
  block_sums<2>(v, red);
  if (threadIdx.x == 0) {
    partial[blockIdx.x] = v[0];
    partial[gridDim.x + blockIdx.x] = v[1];
  }
  if (last_block(counter)) {
    block_final_sums<2>(gridDim.x, partial, gridDim.x, v, red);
    if (threadIdx.x == 0) {
      sc[S_NUM] = v[0];
      sc[S_BETA] = v[0] / sc[S_RZ];
      sc[S_RZN] = v[1];
      sc[S_RZ] = v[1];
    }
  }
}

// The start of CG, z = MGI(0, r) given: p = z and r.z into sc[S_RZ] (partials,
// finished by the last block).  Grid: kRedBlocks x 256.
template <class Z>
__global__ void __launch_bounds__(256, 4) k_pcg_first(int64_t n, const Z* __restrict__ z, const double* __restrict__ r,
                                                   double* __restrict__ p, double* __restrict__ partial,
                                                   int* counter, double* sc) {
  __shared__ double red[1][256];
  pdl_wait();
  pdl_trigger();
  double rz = 0.0;
#pragma unroll 4
  for (int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x; i < n; i += (int64_t)gridDim.x * 256) {
    const double zi = to_f64(z[i]);
    p[i] = zi;
    rz += r[i] * zi;
  }
  double v[1] = {rz};
  block_sums<1>(v, red);
  if (threadIdx.x == 0) partial[blockIdx.x] = v[0];
  if (last_block(counter)) {
    block_final_sums<1>(gridDim.x, partial, 0, v, red);
    if (threadIdx.x == 0) sc[S_RZ] = v[0];
  }
}

// p = z + beta p.
template <class Z>
__global__ void k_pcg_dir(int64_t n, const double* sc, const Z* __restrict__ z, double* __restrict__ p) {
  pdl_wait();
  pdl_trigger();
  const double beta = sc[S_BETA];
  GRID_LOOP(i, n) p[i] = to_f64(z[i]) + beta * p[i];
}
// z = 0 with the rows of colour 0 (the first n0) at their first Gauss-Seidel
// update from zero, (r - 0) / a_ii: the start of an FP64 correction cycle
// MGI(0, r) that reads r as its right-hand side.
__global__ void k_zero_c0(int64_t n, const double* r, double* z, const double* __restrict__ dinv, int64_t n0) {
  pdl_wait();
  pdl_trigger();
  GRID_LOOP(i, n) z[i] = i < n0 ? (r[i] - 0.0) * dinv[i] : 0.0;
}

// ------------------------------------------------------------------ launchers

// Timing events: inside a stream capture they become external event nodes
// of the graph; outside, plain records.
static cudaError_t record_timing_event(cudaEvent_t e, cudaStream_t s) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  cudaError_t err = cudaStreamIsCapturing(s, &cs);
  if (err != cudaSuccess) return err;
  return cs == cudaStreamCaptureStatusActive ? cudaEventRecordWithFlags(e, s, cudaEventRecordExternal)
                                             : cudaEventRecord(e, s);
}

static inline int64_t blocks_for(int64_t threads, int per = 256, int64_t cap = 152 * 64) {
  const int64_t g = (threads + per - 1) / per;
  return std::max<int64_t>(1, std::min<int64_t>(g, cap));
}

template <class T>
gmg_status launch_gs_colour(Level& L, int colour, const T* b, T* x, cudaStream_t s) {
  const int64_t s0 = L.color_slice_off[colour], s1 = L.color_slice_off[colour + 1];
  if (s1 <= s0) return GMG_OK;
  const int G = L.lanes;
  const int64_t grid = (s1 - s0 + (8 / G) - 1) / (8 / G);
  const Ell& A = L.A;
  switch (G) {
    case 1: return launch(k_gs<T, 1>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::dinv(L), b, x);
    case 2: return launch(k_gs<T, 2>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::dinv(L), b, x);
    case 4: return launch(k_gs<T, 4>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::dinv(L), b, x);
    default: return launch(k_gs<T, 8>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::dinv(L), b, x);
  }
}

template <class T, bool NORM>
static gmg_status launch_residual_n(Level& L, const T* x, const T* b, T* r, const NormEnd& end, cudaStream_t s) {
  const int G = L.rlanes;
  int64_t grid = (L.A.nslice + (8 / G) - 1) / (8 / G);
  if (NORM) grid = std::min<int64_t>(grid, kRedBlocks);  // one reduction per resident block
  const Ell& A = L.A;
  switch (G) {
    case 1: return launch(k_residual<T, 1, NORM>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::diag(L), x, b, r, end);
    case 2: return launch(k_residual<T, 2, NORM>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::diag(L), x, b, r, end);
    case 4: return launch(k_residual<T, 4, NORM>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::diag(L), x, b, r, end);
    default: return launch(k_residual<T, 8, NORM>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, Vec<T>::v(A), Vec<T>::diag(L), x, b, r, end);
  }
}

template <class T>
gmg_status launch_residual(Level& L, const T* x, const T* b, T* r, cudaStream_t s) {
  return launch_residual_n<T, false>(L, x, b, r, NormEnd{}, s);
}

template <class T>
gmg_status launch_restrict(Level& L, const T* r, T* bc, T* xc, cudaStream_t s, const T* dinvc, int64_t nc0) {
  const Ell& R = L.R;
  return launch(k_restrict<T>, blocks_for(R.nslice * 32, 256, INT32_MAX), 256, s, R.nslice, R.ptr, R.row0, R.nrow,
                R.col, Vec<T>::v(R), r, bc, xc, dinvc, nc0);
}

template <class T>
gmg_status launch_prolong(Level& L, const T* u, T* x, cudaStream_t s) {
  return launch(k_prolong<T>, blocks_for(L.n, 256, INT32_MAX), 256, s, L.n, L.p_idx, Vec<T>::pw(L), u, x);
}

template <class T>
gmg_status launch_coarse(gmg_ctx* c, const T* b, T* x, cudaStream_t s) {
  const int n = (int)c->nco;
  return launch(k_coarse<T>, (n * 32 + 255) / 256, 256, s, n, (const double*)c->Ainv, b, x);
}

// First level of the cluster form of the cycle in this precision (-1: none).
template <class T>
static int cluster_l0(const gmg_ctx* c) {
  return sizeof(T) == 4 ? c->cl32.l0 : c->cl64.l0;
}

// MGI(x_l, b_l, l) of Alg. 2 on the level's own vectors.  x_l holds the
// initial iterate (zero for every l > 0: the restriction clears it).  With
// c0_done the kernel that produced b_l has already applied the first
// Gauss-Seidel colour to x_l = 0 (the restriction does so for every level it
// feeds that is smoothed), and the first sweep starts at colour 1.
template <class T>
gmg_status vcycle(gmg_ctx* c, int l, cudaStream_t s, bool c0_done, T* x_in, const T* b_in) {
  Level& L = c->L[l];
  T* x = x_in ? x_in : Vec<T>::x(L);
  const T* b = b_in ? b_in : Vec<T>::b(L);
  const bool lp = c->prof && (int)c->lev_ev.size() >= 6 * c->nlev;  // per-level events
  cudaEvent_t* E = lp ? &c->lev_ev[6 * l] : nullptr;
  if (l == c->nlev - 1 || l == cluster_l0<T>(c)) {  // the coarsest solve, or the cluster from this level down
    if (c->inv_pending) {  // a refresh's coarsest inverse may still be running: wait for it here
      cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
      GMG_CK(cudaStreamIsCapturing(s, &cs));
      if (cs != cudaStreamCaptureStatusNone) {
        set_error("internal: coarsest inverse pending during a graph capture");
        return GMG_ERR_CUDA;
      }
      GMG_TRY(join_inverse(c, s, false));
    }
    if (lp) {
      GMG_CK(record_timing_event(E[0], s));
      c->lev_kind[l] = 2;
      c->lev_gs[l] = 0;
    }
    if (c->prof && l == 0)  // no finest smoothing blocks of their own: an empty interval before and after
      for (int q : {0, 1}) GMG_CK(record_timing_event(c->ev[q], s));
    if (l == c->nlev - 1) GMG_TRY(launch_coarse<T>(c, b, x, s));
    else GMG_TRY(launch_cluster<T>(c, x, b, c0_done, s));
    if (c->prof && l == 0) {
      for (int q : {2, 3}) GMG_CK(record_timing_event(c->ev[q], s));
      c->prof_gs = 0;
    }
    if (lp) {
      GMG_CK(record_timing_event(E[5], s));
      for (int k = l + 1; k < c->nlev; ++k) c->lev_kind[k] = 0;
    }
    return GMG_OK;
  }
  Level& C = c->L[l + 1];
  const bool prof = c->prof && l == 0;
  if (prof) GMG_CK(record_timing_event(c->ev[0], s));
  if (lp) GMG_CK(record_timing_event(E[0], s));
  int gs = 0;
  for (int it = 0; it < c->opt.nu_pre; ++it)
    for (int k = (it == 0 && c0_done) ? 1 : 0; k < L.ncolor; ++k, ++gs) GMG_TRY(launch_gs_colour<T>(L, k, b, x, s));
  if (prof) GMG_CK(record_timing_event(c->ev[1], s));
  if (lp) GMG_CK(record_timing_event(E[1], s));
  GMG_TRY(launch_residual<T>(L, x, b, Vec<T>::r(L), s));
  const bool next_c0 = c->opt.nu_pre > 0 && l + 1 < c->nlev - 1;
  GMG_TRY(launch_restrict<T>(L, Vec<T>::r(L), Vec<T>::b(C), Vec<T>::x(C), s, next_c0 ? Vec<T>::dinv(C) : nullptr,
                             next_c0 ? C.color_off[1] : 0));
  if (lp) GMG_CK(record_timing_event(E[2], s));
  GMG_TRY(vcycle<T>(c, l + 1, s, next_c0));
  if (lp) GMG_CK(record_timing_event(E[3], s));
  GMG_TRY(launch_prolong<T>(L, Vec<T>::x(C), x, s));
  if (prof) GMG_CK(record_timing_event(c->ev[2], s));
  if (lp) GMG_CK(record_timing_event(E[4], s));
  for (int it = 0; it < c->opt.nu_post; ++it)
    for (int q = 0; q < L.ncolor; ++q, ++gs) {
      const int k = c->opt.post_forward ? q : L.ncolor - 1 - q;
      GMG_TRY(launch_gs_colour<T>(L, k, b, x, s));
    }
  if (prof) {
    GMG_CK(record_timing_event(c->ev[3], s));
    c->prof_gs = gs;
  }
  if (lp) {
    GMG_CK(record_timing_event(E[5], s));
    c->lev_kind[l] = 1;
    c->lev_gs[l] = gs;
  }
  return GMG_OK;
}

template gmg_status launch_gs_colour<double>(Level&, int, const double*, double*, cudaStream_t);
template gmg_status launch_gs_colour<float>(Level&, int, const float*, float*, cudaStream_t);
template gmg_status launch_residual<double>(Level&, const double*, const double*, double*, cudaStream_t);
template gmg_status launch_residual<float>(Level&, const float*, const float*, float*, cudaStream_t);
template gmg_status launch_restrict<double>(Level&, const double*, double*, double*, cudaStream_t, const double*,
                                           int64_t);
template gmg_status launch_restrict<float>(Level&, const float*, float*, float*, cudaStream_t, const float*, int64_t);
template gmg_status launch_prolong<double>(Level&, const double*, double*, cudaStream_t);
template gmg_status launch_prolong<float>(Level&, const float*, float*, cudaStream_t);
template gmg_status launch_coarse<double>(gmg_ctx*, const double*, double*, cudaStream_t);
template gmg_status launch_coarse<float>(gmg_ctx*, const float*, float*, cudaStream_t);
template gmg_status vcycle<double>(gmg_ctx*, int, cudaStream_t, bool, double*, const double*);
template gmg_status vcycle<float>(gmg_ctx*, int, cudaStream_t, bool, float*, const float*);

gmg_status launch_gather(int64_t n, const int32_t* perm, const double* src, double* dst, cudaStream_t s) {
  return launch(k_gather, blocks_for(n), 256, s, n, perm, src, dst);
}
gmg_status launch_scatter_cycle(gmg_ctx* c, const double* src, double* dst, cudaStream_t s) {
  Level& L = c->L[0];
  return launch(k_scatter_cycle, blocks_for(L.n), 256, s, L.n, L.perm, src, dst, (const int*)(c->dstatus + 3));
}
gmg_status launch_scatter(int64_t n, const int32_t* perm, const double* src, double* dst, cudaStream_t s) {
  return launch(k_scatter_vec, blocks_for(n), 256, s, n, perm, src, dst);
}
gmg_status launch_d2f(int64_t n, const double* a, float* b, cudaStream_t s) {
  return launch(k_d2f, blocks_for(n), 256, s, n, a, b);
}
gmg_status launch_f2d(int64_t n, const float* a, double* b, cudaStream_t s) {
  return launch(k_f2d, blocks_for(n), 256, s, n, a, b);
}

// ------------------------------------------------------------------ outer iteration

// rs = bs - A xs (FP64, finest level) and sc[S_RR] = ||rs||^2, then `what`
// (kNorm*) with the loop condition h.
static gmg_status outer_residual(gmg_ctx* c, int what, cudaStream_t s, cudaGraphConditionalHandle h = 0) {
  Level& L = c->L[0];
  const NormEnd end{c->red, c->red_cnt + 4, c->scal, c->dloop, c->dhist, h, what};
  return launch_residual_n<double, true>(L, c->xs, c->bs, c->rs, end, s);
}

// A finest-level V-cycle, bracketed by timing events when profiling is on;
// x and b replace the finest level's own vectors when given.
template <class T>
static gmg_status timed_vcycle(gmg_ctx* c, cudaStream_t s, bool c0_done, T* x = nullptr, const T* b = nullptr) {
  if (c->prof) GMG_CK(record_timing_event(c->ev[4], s));
  GMG_TRY(vcycle<T>(c, 0, s, c0_done, x, b));
  if (c->prof) GMG_CK(record_timing_event(c->ev[5], s));
  return GMG_OK;
}

static bool pcg_mode(int mode) { return mode == GMG_FP32_PCG || mode == GMG_FP64_PCG; }

// One outer iteration (captured as a graph when enabled).
//  FP64         : x <- MGI(x, b) (FP64 cycle on the iterate), r = b - A x, rr
//  FP32_REFINE  : e = MGI32(0, r), x += e, r = b - A x, rr
//  *_PCG seg 0  : q = A p, pq, alpha = rz/pq, x += alpha p, r -= alpha q, rr
//  *_PCG seg 1  : z = MGI(0, r) (FP32 or FP64 cycle), num = z.(r - r_old),
//                 rz' = r.z, p = z + (num/rz) p, rz = rz'
gmg_status iteration_body(gmg_ctx* c, int mode, int seg, cudaStream_t s, cudaGraphConditionalHandle h, bool check) {
  Level& L = c->L[0];
  const int64_t n = L.n;
  const int64_t n0 = c->opt.nu_pre > 0 ? L.color_off[1] : 0;
  if (mode == GMG_FP64) {
    GMG_TRY(timed_vcycle<double>(c, s, false));  // level-0 x64/b64 alias xs/bs
    return outer_residual(c, check ? kNormIter : kNormOnly, s, h);
  }
  if (mode == GMG_FP32_REFINE) {
    GMG_TRY(launch(k_d2f_zero, blocks_for(n), 256, s, n, (const double*)c->rs, L.b32, L.x32, (const float*)L.dinv32,
                   n0));
    GMG_TRY(timed_vcycle<float>(c, s, n0 > 0));
    GMG_TRY(launch(k_add_f2d, blocks_for(n), 256, s, n, (const float*)L.x32, c->xs));
    return outer_residual(c, check ? kNormIter : kNormOnly, s, h);
  }
  const bool f64 = mode == GMG_FP64_PCG;
  if (seg == 0) {
    const int64_t nb = std::min<int64_t>((L.A.nslice + 7) / 8, kRedBlocks);  // one reduction per resident block
    GMG_TRY(launch(k_spmv_dot, nb, 256, s, L.A.nslice, L.A.ptr, L.A.row0, L.A.nrow, L.A.col, L.A.v64, L.diag64,
                   (const double*)c->ps, c->qs, c->red, c->red_cnt, c->scal + S_PQ));
    if (f64)
      return launch(k_pcg_axpy<double>, kRedBlocks, 256, s, n, c->scal, (const double*)c->ps, (const double*)c->qs,
                    c->xs, c->rs, c->ros, (float*)nullptr, c->zs, (const double*)L.dinv64, n0, c->red,
                    c->red_cnt + 1, check ? 1 : 0, c->dloop, c->dhist, h);
    return launch(k_pcg_axpy<float>, kRedBlocks, 256, s, n, c->scal, (const double*)c->ps, (const double*)c->qs,
                  c->xs, c->rs, c->ros, L.b32, L.x32, (const float*)L.dinv32, n0, c->red, c->red_cnt + 1,
                  check ? 1 : 0, c->dloop, c->dhist, h);
  }
  // the cycle's right-hand side and initial iterate (colour 0 already
  // smoothed from zero) were set by segment 0
  if (f64) {
    GMG_TRY(timed_vcycle<double>(c, s, n0 > 0, c->zs, (const double*)c->rs));
    GMG_TRY(launch(k_pcg_zdots<double>, kRedBlocks, 256, s, n, (const double*)c->zs, (const double*)c->rs,
                   (const double*)c->ros, c->red, c->red_cnt + 2, c->scal));
    return launch(k_pcg_dir<double>, blocks_for(n), 256, s, n, (const double*)c->scal, (const double*)c->zs, c->ps);
  }
  GMG_TRY(timed_vcycle<float>(c, s, n0 > 0));
  GMG_TRY(launch(k_pcg_zdots<float>, kRedBlocks, 256, s, n, (const float*)L.x32, (const double*)c->rs,
                 (const double*)c->ros, c->red, c->red_cnt + 2, c->scal));
  return launch(k_pcg_dir<float>, blocks_for(n), 256, s, n, (const double*)c->scal, (const float*)L.x32, c->ps);
}

// PCG start: z = MGI(0, r) in the mode's cycle precision (FP64: zs is the
// cycle's iterate, FP32: the finest level's x32), rz = r.z, p = z (r must be
// current).
gmg_status pcg_start(gmg_ctx* c, int mode, cudaStream_t s) {
  Level& L = c->L[0];
  const int64_t n = L.n, n0 = c->opt.nu_pre > 0 ? L.color_off[1] : 0;
  const double* r = c->rs;
  if (mode == GMG_FP64_PCG) {
    GMG_TRY(launch(k_zero_c0, blocks_for(n), 256, s, n, r, c->zs, (const double*)L.dinv64, n0));
    GMG_TRY(timed_vcycle<double>(c, s, n0 > 0, c->zs, r));
    return launch(k_pcg_first<double>, kRedBlocks, 256, s, n, (const double*)c->zs, r, c->ps, c->red, c->red_cnt + 2,
                  c->scal);
  }
  GMG_TRY(launch(k_d2f_zero, blocks_for(n), 256, s, n, r, L.b32, L.x32, (const float*)L.dinv32, n0));
  GMG_TRY(timed_vcycle<float>(c, s, n0 > 0));
  return launch(k_pcg_first<float>, kRedBlocks, 256, s, n, (const float*)L.x32, r, c->ps, c->red, c->red_cnt + 2,
                c->scal);
}

gmg_status loop_body(gmg_ctx* c, int mode, cudaGraphConditionalHandle h, cudaStream_t s) {
  if (pcg_mode(mode)) GMG_TRY(iteration_body(c, mode, 1, s));
  return iteration_body(c, mode, 0, s, h, true);
}

gmg_status outer_residual_norm(gmg_ctx* c, bool start, cudaStream_t s) {
  return outer_residual(c, start ? kNormStart : kNormOnly, s);
}

gmg_status load_system(gmg_ctx* c, const double* b, const double* x, double tol, cudaStream_t s) {
  Level& L = c->L[0];
  return launch(k_load, kRedBlocks, 256, s, L.n, L.perm, b, x, c->bs, c->xs, c->red, c->red_cnt + 5, c->scal, c->dloop,
                tol, c->opt.max_iter, c->dstatus + 3);
}

gmg_status store_solution(gmg_ctx* c, double* x, cudaStream_t s) {
  Level& L = c->L[0];
  return launch(k_store, blocks_for(L.n), 256, s, L.n, L.perm, (const double*)c->xs, x, (const double*)c->scal,
                (const int*)c->dloop, (const double*)c->dhist, (const int*)c->dstatus, c->h_scal);
}

}  // namespace gmg
