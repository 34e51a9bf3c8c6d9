// Many right-hand sides at once (SpMM-style V-cycle): every level's vectors
// are [n_l x NR] row-major in the permuted numbering, so each matrix entry is
// read once and applied to NR contiguous values (NR = 1, 2, 4, 8 or 16; the
// caller's nrhs is padded with zero columns).  The inner cycle runs in FP32
// (coarsest solve in FP64) inside FP64 iterative refinement, as in Alg. 1
// with the correction form x += MGI(0, b - A x).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <string>

#include "gmg_cycle.cuh"

namespace gmg {

// Columns of a block are split over Q lanes of V columns each (NR = 1, 2: one
// lane; 4, 8, 16: one, two, four lanes of a float4), so that the lanes of a
// row read and write its NR values as one contiguous piece and 32 / Q rows
// share a warp.
template <int NR>
struct MCols {
  static constexpr int V = NR < 4 ? NR : 4;
  static constexpr int Q = NR / V;
};
// Entries of a row part whose gathers are in flight together (131,072 rows x 8
// columns: 4.14 ms a solve, 4.56 with four).
constexpr int kMPre = 8;
// Warps per coarse row in the restriction (18-40 terms per row): 4.20, 4.17,
// 4.14 and 4.21 ms for the same solve with 1, 2, 4 and 8.
constexpr int kMRestrictParts = 4;

template <int V>
__device__ __forceinline__ void load_cols(const float* p, float (&o)[V]) {
  if constexpr (V == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    o[0] = q.x;
    o[1] = q.y;
    o[2] = q.z;
    o[3] = q.w;
  } else if constexpr (V == 2) {
    const float2 q = *reinterpret_cast<const float2*>(p);
    o[0] = q.x;
    o[1] = q.y;
  } else {
    o[0] = *p;
  }
}
template <int V>
__device__ __forceinline__ void store_cols(float* p, const float (&o)[V]) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(p) = make_float4(o[0], o[1], o[2], o[3]);
  else if constexpr (V == 2) *reinterpret_cast<float2*>(p) = make_float2(o[0], o[1]);
  else *p = o[0];
}

// One lane's share of a row: row group `group` (32 / Q rows of one slice),
// warp `part` of the G that split its entries.  The first kMPre values and
// columns are loaded here, before the dependency wait.
template <int NR, int G>
struct MRow {
  bool active;
  int nk, c;    // entries of this part, first column of this lane
  int64_t e, r;
  float v[kMPre];
  int32_t j[kMPre];
  __device__ __forceinline__ MRow(int64_t s0, int64_t s1, int64_t group, const int64_t* __restrict__ ptr,
                                  const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                  const int32_t* __restrict__ col, const float* __restrict__ val, int part, int lane) {
    constexpr int Q = MCols<NR>::Q;
    const int64_t s = s0 + group / Q;
    const int ri = (int)(group % Q) * (32 / Q) + lane / Q;
    active = false;
    nk = 0;
    c = (lane % Q) * MCols<NR>::V;
    e = r = 0;
    if (s < s1) {
      active = ri < nrow[s];
      const int64_t e0 = ptr[s];
      const int w = (int)((ptr[s + 1] - e0) >> 5);
      nk = active && part < w ? (w - part + G - 1) / G : 0;
      e = e0 + (int64_t)part * 32 + ri;
      r = row0[s] + ri;
    }
#pragma unroll
    for (int q = 0; q < kMPre; ++q) {
      v[q] = q < nk ? val[e + (int64_t)q * G * 32] : 0.f;
      j[q] = q < nk ? col[e + (int64_t)q * G * 32] : 0;
    }
  }
  // acc[c] += sum over this part's entries of a_rk X[k][c], entries in order;
  // the gathers of kMPre entries are issued together (one after another, as
  // a loop over the entries, a coarse colour took 10.5 us)
  __device__ __forceinline__ void dot(const int32_t* __restrict__ col, const float* __restrict__ val, const float* X,
                                      float (&acc)[MCols<NR>::V]) {
    constexpr int V = MCols<NR>::V;
    for (int q0 = 0; q0 < nk; q0 += kMPre) {
      float xv[kMPre][V];
#pragma unroll
      for (int q = 0; q < kMPre; ++q)
        if (q0 + q < nk) load_cols<V>(X + (int64_t)j[q] * NR + c, xv[q]);
#pragma unroll
      for (int q = 0; q < kMPre; ++q)
        if (q0 + q < nk)
#pragma unroll
          for (int k = 0; k < V; ++k) acc[k] += v[q] * xv[q][k];
      if (q0 + kMPre < nk)
#pragma unroll
        for (int q = 0; q < kMPre; ++q) {
          const bool in = q0 + kMPre + q < nk;
          v[q] = in ? val[e + (int64_t)(q0 + kMPre + q) * G * 32] : 0.f;
          j[q] = in ? col[e + (int64_t)(q0 + kMPre + q) * G * 32] : 0;
        }
    }
  }
};

// Adds the other G - 1 warps' partial sums to row part 0's, in warp order.
template <int V, int G>
__device__ __forceinline__ void m_combine(float (&acc)[V], int warp, int lane) {
  if constexpr (G > 1) {
    __shared__ float red[8][V][32];
#pragma unroll
    for (int c = 0; c < V; ++c) red[warp][c][lane] = acc[c];
    __syncthreads();
    if (warp % G == 0)
#pragma unroll
      for (int g = 1; g < G; ++g)
#pragma unroll
        for (int c = 0; c < V; ++c) acc[c] += red[warp + g][c][lane];
  }
}

// One colour of a multi-right-hand-side Gauss-Seidel sweep, rows split over G warps.
template <int NR, int G>
__global__ void __launch_bounds__(256) k_gs_m(int64_t s0, int64_t s1, const int64_t* __restrict__ ptr,
                                              const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                              const int32_t* __restrict__ col, const float* __restrict__ val,
                                              const float* __restrict__ dinv, const float* B, float* X) {
  constexpr int V = MCols<NR>::V;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % G;
  MRow<NR, G> m(s0, s1, (int64_t)blockIdx.x * (8 / G) + warp / G, ptr, row0, nrow, col, val, part, lane);
  const bool own = part == 0 && m.active;
  const float d = own ? dinv[m.r] : 0.f;
  pdl_wait();
  pdl_trigger();
  float acc[V], bv[V];
#pragma unroll
  for (int c = 0; c < V; ++c) acc[c] = bv[c] = 0.f;
  if (own) load_cols<V>(B + m.r * NR + m.c, bv);  // issued with the gathers, not after the combining barrier
  m.dot(col, val, X, acc);                        // other colours: not written by this launch
  m_combine<V, G>(acc, warp, lane);
  if (own) {
#pragma unroll
    for (int c = 0; c < V; ++c) acc[c] = (bv[c] - acc[c]) * d;
    store_cols<V>(X + m.r * NR + m.c, acc);
  }
}

// R = B - A X over all slices, rows split over G warps.
template <int NR, int G>
__global__ void __launch_bounds__(256) k_residual_m(int64_t nslice, const int64_t* __restrict__ ptr,
                                                    const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                                    const int32_t* __restrict__ col, const float* __restrict__ val,
                                                    const float* __restrict__ diag, const float* X, const float* B,
                                                    float* R) {
  constexpr int V = MCols<NR>::V;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % G;
  MRow<NR, G> m(0, nslice, (int64_t)blockIdx.x * (8 / G) + warp / G, ptr, row0, nrow, col, val, part, lane);
  const bool own = part == 0 && m.active;
  const float d = own ? diag[m.r] : 0.f;
  pdl_wait();
  pdl_trigger();
  float acc[V], bv[V];
#pragma unroll
  for (int c = 0; c < V; ++c) acc[c] = bv[c] = 0.f;
  if (own) {
    load_cols<V>(X + m.r * NR + m.c, acc);
    load_cols<V>(B + m.r * NR + m.c, bv);
#pragma unroll
    for (int c = 0; c < V; ++c) acc[c] *= d;
  }
  m.dot(col, val, X, acc);
  m_combine<V, G>(acc, warp, lane);
  if (own) {
#pragma unroll
    for (int c = 0; c < V; ++c) acc[c] = bv[c] - acc[c];
    store_cols<V>(R + m.r * NR + m.c, acc);
  }
}

// Bc = P^T R; the coarse iterate Xc starts from zero, but its rows of colour 0
// (the first nc0) take their first Gauss-Seidel update (b - 0) / a_ii.
template <int NR>
__global__ void __launch_bounds__(256) k_restrict_m(int64_t nslice, const int64_t* __restrict__ ptr,
                                                    const int32_t* __restrict__ row0, const int32_t* __restrict__ nrow,
                                                    const int32_t* __restrict__ col, const float* __restrict__ w,
                                                    const float* R, float* Bc, float* Xc,
                                                    const float* __restrict__ dinvc, int64_t nc0) {
  constexpr int V = MCols<NR>::V, G = kMRestrictParts;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, part = warp % G;
  MRow<NR, G> m(0, nslice, (int64_t)blockIdx.x * (8 / G) + warp / G, ptr, row0, nrow, col, w, part, lane);
  const bool own = part == 0 && m.active;
  const float d = own && m.r < nc0 ? dinvc[m.r] : 0.f;
  pdl_wait();
  pdl_trigger();
  float acc[V];
#pragma unroll
  for (int c = 0; c < V; ++c) acc[c] = 0.f;
  m.dot(col, w, R, acc);
  m_combine<V, G>(acc, warp, lane);
  if (own) {
    store_cols<V>(Bc + m.r * NR + m.c, acc);
#pragma unroll
    for (int c = 0; c < V; ++c) acc[c] = m.r < nc0 ? (acc[c] - 0.f) * d : 0.f;
    store_cols<V>(Xc + m.r * NR + m.c, acc);
  }
}

// X += P U, one thread per row and column group.
template <int NR>
__global__ void __launch_bounds__(256) k_prolong_m(int64_t n, const int32_t* __restrict__ idx,
                                                   const float* __restrict__ w, const float* U, float* X) {
  constexpr int V = MCols<NR>::V, Q = MCols<NR>::Q;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, i = t / Q;
  const int c0 = (int)(t % Q) * V;
  int32_t id[3] = {0, 0, 0};
  float a[3] = {0.f, 0.f, 0.f};
  if (i < n)
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      id[m] = idx[3 * i + m];
      a[m] = w[3 * i + m];
    }
  pdl_wait();
  pdl_trigger();
  if (i >= n) return;
  float xv[V], u[3][V];
  load_cols<V>(X + i * NR + c0, xv);
#pragma unroll
  for (int m = 0; m < 3; ++m) load_cols<V>(U + (int64_t)id[m] * NR + c0, u[m]);
#pragma unroll
  for (int m = 0; m < 3; ++m)
#pragma unroll
    for (int c = 0; c < V; ++c) xv[c] += a[m] * u[m][c];
  store_cols<V>(X + i * NR + c0, xv);
}

// X = Ainv B on the coarsest level (FP64 accumulation), one warp per row and
// pair of columns: the FP64 pipes bound it (a warp instruction occupies a
// sub-partition's pipe for 64 cycles), so the work is spread over all of them.
template <int NR>
__global__ void __launch_bounds__(256) k_coarse_m(int n, const double* __restrict__ Ainv, const float* B, float* X) {
  constexpr int W = NR < 2 ? 1 : 2;
  const int t = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  const int row = t / (NR / W), c0 = (t % (NR / W)) * W;
  pdl_wait();
  pdl_trigger();
  if (row >= n) return;
  double s[W];
#pragma unroll
  for (int c = 0; c < W; ++c) s[c] = 0.0;
  const double* a = Ainv + (int64_t)row * n;
#pragma unroll 4
  for (int j = lane; j < n; j += 32) {
    const double aj = a[j];
    float bv[W];
    load_cols<W>(B + (int64_t)j * NR + c0, bv);
#pragma unroll
    for (int c = 0; c < W; ++c) s[c] += aj * f64_of(bv[c]);
  }
#pragma unroll
  for (int c = 0; c < W; ++c)
    for (int o = 16; o > 0; o >>= 1) s[c] += __shfl_xor_sync(0xffffffffu, s[c], o);
  if (lane == 0) {
    float xv[W];
#pragma unroll
    for (int c = 0; c < W; ++c) xv[c] = f32_rn(s[c]);
    store_cols<W>(X + (int64_t)row * NR + c0, xv);
  }
}

// FP64 outer residual R = B - A X, one lane per row and pair of columns
// (32 / Q rows per warp), a fixed grid walking the row groups: the correction
// cycle's right-hand side R32 = (float) R and initial iterate X32 (zero, the
// rows of colour 0, the first n0, at their first Gauss-Seidel update), and the
// columns' sums of R^2 into out[0 .. NR) (block partials, finished in a fixed
// order by the last block).
template <int NR>
__global__ void __launch_bounds__(256) k_outer_residual_m(int64_t nslice, const int64_t* __restrict__ ptr,
                                                          const int32_t* __restrict__ row0,
                                                          const int32_t* __restrict__ nrow,
                                                          const int32_t* __restrict__ col,
                                                          const double* __restrict__ val,
                                                          const double* __restrict__ diag, const double* X,
                                                          const double* B, float* R32, float* X32,
                                                          const float* __restrict__ dinv32, int64_t n0,
                                                          double* partial, int* counter, double* out) {
  constexpr int V = NR < 2 ? 1 : 2, Q = NR / V, RW = 32 / Q, U = 4;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = (lane % Q) * V;
  pdl_wait();
  pdl_trigger();
  double sq[V];
#pragma unroll
  for (int c = 0; c < V; ++c) sq[c] = 0.0;
  for (int64_t g = (int64_t)blockIdx.x * 8 + warp; g < nslice * Q; g += (int64_t)gridDim.x * 8) {
    const int64_t s = g / Q;
    const int ri = (int)(g % Q) * RW + lane / Q;
    if (ri >= nrow[s]) continue;
    const int64_t r = row0[s] + ri, e = ptr[s] + ri;
    const int w = (int)((ptr[s + 1] - ptr[s]) >> 5);
    double acc[V], bv[V];
    const double d = diag[r];
#pragma unroll
    for (int c = 0; c < V; ++c) {
      acc[c] = d * X[r * NR + c0 + c];
      bv[c] = B[r * NR + c0 + c];
    }
    for (int k0 = 0; k0 < w; k0 += U) {
      double a[U], xv[U][V];
      int32_t j[U];
#pragma unroll
      for (int q = 0; q < U; ++q) {
        a[q] = k0 + q < w ? val[e + (int64_t)(k0 + q) * 32] : 0.0;
        j[q] = k0 + q < w ? col[e + (int64_t)(k0 + q) * 32] : (int32_t)r;
      }
#pragma unroll
      for (int q = 0; q < U; ++q)
        if constexpr (V == 2) {
          const double2 t = *reinterpret_cast<const double2*>(X + (int64_t)j[q] * NR + c0);
          xv[q][0] = t.x;
          xv[q][1] = t.y;
        } else {
          xv[q][0] = X[(int64_t)j[q] * NR + c0];
        }
#pragma unroll
      for (int q = 0; q < U; ++q)
        if (k0 + q < w)
#pragma unroll
          for (int c = 0; c < V; ++c) acc[c] += a[q] * xv[q][c];
    }
    const float di = r < n0 ? dinv32[r] : 0.f;
    float rv32[V], xv32[V];
#pragma unroll
    for (int c = 0; c < V; ++c) {
      const double rv = bv[c] - acc[c];
      sq[c] += rv * rv;
      rv32[c] = f32_rn(rv);
      xv32[c] = r < n0 ? (rv32[c] - 0.f) * di : 0.f;
    }
    store_cols<V>(R32 + r * NR + c0, rv32);
    store_cols<V>(X32 + r * NR + c0, xv32);
  }
  // sums over the block's rows: lanes of a column group, then the warps in order
  __shared__ double red[8][NR];
#pragma unroll
  for (int c = 0; c < V; ++c)
    for (int o = 16; o >= Q; o >>= 1) sq[c] += __shfl_xor_sync(0xffffffffu, sq[c], o);
  if (lane < Q)
#pragma unroll
    for (int c = 0; c < V; ++c) red[warp][c0 + c] = sq[c];
  __syncthreads();
  if (threadIdx.x < NR) {
    double t = 0.0;
    for (int q = 0; q < 8; ++q) t += red[q][threadIdx.x];
    partial[(int64_t)blockIdx.x * NR + threadIdx.x] = t;
  }
  __shared__ int is_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    is_last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
    if (is_last) *counter = 0;
  }
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  for (int c = warp; c < NR; c += 8) {  // a warp per column
    double t = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(partial + (int64_t)b * NR + c);
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) out[c] = t;
  }
}

// Caller [n x nrhs] (double) -> permuted [n x NR] with zero padding, and back.
__global__ void k_gather_m(int64_t n, int nrhs, int NR, const int32_t* __restrict__ perm, const double* __restrict__ src,
                           double* __restrict__ dst) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * NR; t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / NR;
    const int c = (int)(t % NR);
    dst[t] = c < nrhs ? src[(int64_t)perm[i] * nrhs + c] : 0.0;
  }
}
__global__ void k_scatter_m(int64_t n, int nrhs, int NR, const int32_t* __restrict__ perm,
                            const double* __restrict__ src, double* __restrict__ dst) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * nrhs;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / nrhs;
    const int c = (int)(t % nrhs);
    dst[(int64_t)perm[i] * nrhs + c] = src[i * NR + c];
  }
}
__global__ void k_zero_cols(int64_t n, int NR, int mask, double* __restrict__ X) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * NR; t += (int64_t)gridDim.x * blockDim.x)
    if ((mask >> (int)(t % NR)) & 1) X[t] = 0.0;
}
// x += (double) e, four consecutive values per thread.
__global__ void __launch_bounds__(256) k_add_f2d_m(int64_t m, const float* e, double* x) {
  pdl_wait();
  pdl_trigger();
  for (int64_t i = 4 * ((int64_t)blockIdx.x * blockDim.x + threadIdx.x); i < m; i += 4 * (int64_t)gridDim.x * blockDim.x) {
    if (i + 4 <= m) {
      const float4 q = *reinterpret_cast<const float4*>(e + i);
      double2* p = reinterpret_cast<double2*>(x + i);
      double2 a = p[0], b = p[1];
      a.x += f64_of(q.x);
      a.y += f64_of(q.y);
      b.x += f64_of(q.z);
      b.y += f64_of(q.w);
      p[0] = a;
      p[1] = b;
    } else {
      for (int64_t k = i; k < m; ++k) x[k] += f64_of(e[k]);
    }
  }
}
// After an iteration of the batched solve (one warp): the worst column's
// relative residual into hist[k] (a non-finite column's value as it is), and
// whether the loop goes on.  it: iterations done, limit, columns; nb: column
// norms of B, finite (0: a zero column).
__global__ void k_batched_check(int* it, double* hist, const double* rr, const double* nb, const double* tol,
                                cudaGraphConditionalHandle h) {
  pdl_wait();
  pdl_trigger();
  const int lane = threadIdx.x;
  const double b = lane < it[2] ? nb[lane] : 0.0;
  const double r = b == 0.0 ? 0.0 : sqrt(rr[lane]) / b;
  const unsigned bad = __ballot_sync(0xffffffffu, !isfinite(r));
  double w = r;
  for (int o = 16; o > 0; o >>= 1) w = fmax(w, __shfl_xor_sync(0xffffffffu, w, o));
  if (bad) w = __shfl_sync(0xffffffffu, r, __ffs(bad) - 1);
  if (lane == 0) {
    const int k = ++it[0];
    hist[k] = w;
    cudaGraphSetConditional(h, !bad && !(w <= *tol) && k < it[1] ? 1u : 0u);
  }
}

static inline int gblk(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 64)); }

#define LCK() GMG_LAUNCHED()

// The warps-per-row split of a level's multi-right-hand-side sweeps and
// residual for NR columns: the autotuned or set choice, else a default by the
// level's mean row length (about 8 entries per warp).
template <int NR>
static int m_lanes(const Level& L) {
  const int v = L.mlanes[nr_index(NR)];
  if (v > 0) return v;
  const double mean = L.n > 0 ? (double)L.nnz / (double)L.n : 1.0;
  return mean <= 12 ? 1 : mean <= 24 ? 2 : mean <= 48 ? 4 : 8;
}

template <int NR>
static gmg_status sweep_m(Level& L, int k, cudaStream_t s, int G = 0) {
  const int64_t s0 = L.color_slice_off[k], s1 = L.color_slice_off[k + 1];
  if (s1 <= s0) return GMG_OK;
  if (G == 0) G = m_lanes<NR>(L);
  const int64_t grid = ((s1 - s0) * MCols<NR>::Q + 8 / G - 1) / (8 / G);
  const Ell& A = L.A;
  const float *v = A.v32, *d = L.dinv32, *b = L.B32;
  switch (G) {
    case 1: return launch(k_gs_m<NR, 1>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, v, d, b, L.X32);
    case 2: return launch(k_gs_m<NR, 2>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, v, d, b, L.X32);
    case 4: return launch(k_gs_m<NR, 4>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, v, d, b, L.X32);
    default: return launch(k_gs_m<NR, 8>, grid, 256, s, s0, s1, A.ptr, A.row0, A.nrow, A.col, v, d, b, L.X32);
  }
}

template <int NR>
static gmg_status residual_m(Level& L, cudaStream_t s, int G = 0) {
  if (G == 0) G = m_lanes<NR>(L);
  const Ell& A = L.A;
  const int64_t grid = (A.nslice * MCols<NR>::Q + 8 / G - 1) / (8 / G);
  const float *v = A.v32, *d = L.diag32, *x = L.X32, *b = L.B32;
  switch (G) {
    case 1: return launch(k_residual_m<NR, 1>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, v, d, x, b, L.R32);
    case 2: return launch(k_residual_m<NR, 2>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, v, d, x, b, L.R32);
    case 4: return launch(k_residual_m<NR, 4>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, v, d, x, b, L.R32);
    default: return launch(k_residual_m<NR, 8>, grid, 256, s, A.nslice, A.ptr, A.row0, A.nrow, A.col, v, d, x, b, L.R32);
  }
}

// MGI(X_l, B_l, l) on [n_l x NR] blocks from the iterate in X_l.  With c0_done
// the kernel that set B_l has set X_l to zero and applied the first
// Gauss-Seidel colour (the outer residual on the finest level, the
// restriction on the others).
template <int NR>
static gmg_status vcycle_m(gmg_ctx* c, int l, cudaStream_t s, bool c0_done) {
  Level& L = c->L[l];
  if (l == c->nlev - 1) {
    constexpr int W = NR < 2 ? 1 : 2;
    return launch(k_coarse_m<NR>, (L.n * (NR / W) * 32 + 255) / 256, 256, s, (int)L.n, (const double*)c->Ainv,
                  (const float*)L.B32, L.X32);
  }
  Level& C = c->L[l + 1];
  for (int it = 0; it < c->opt.nu_pre; ++it)
    for (int k = it == 0 && c0_done ? 1 : 0; k < L.ncolor; ++k) GMG_TRY(sweep_m<NR>(L, k, s));
  GMG_TRY(residual_m<NR>(L, s));
  const bool next_c0 = c->opt.nu_pre > 0 && l + 1 < c->nlev - 1;
  const int64_t rgrid = (L.R.nslice * MCols<NR>::Q + 8 / kMRestrictParts - 1) / (8 / kMRestrictParts);
  GMG_TRY(launch(k_restrict_m<NR>, rgrid, 256, s, L.R.nslice, L.R.ptr, L.R.row0, L.R.nrow, L.R.col, L.R.v32,
                 (const float*)L.R32, C.B32, C.X32, (const float*)C.dinv32, next_c0 ? C.color_off[1] : (int64_t)0));
  GMG_TRY(vcycle_m<NR>(c, l + 1, s, next_c0));
  GMG_TRY(launch(k_prolong_m<NR>, (L.n * MCols<NR>::Q + 255) / 256, 256, s, L.n, L.p_idx, L.p_w32,
                 (const float*)C.X32, L.X32));
  for (int it = 0; it < c->opt.nu_post; ++it)
    for (int q = 0; q < L.ncolor; ++q) GMG_TRY(sweep_m<NR>(L, c->opt.post_forward ? q : L.ncolor - 1 - q, s));
  return GMG_OK;
}

// Rows of the finest level whose first update the outer residual applies.
static int64_t first_rows(const gmg_ctx* c) { return c->opt.nu_pre > 0 && c->nlev > 1 ? c->L[0].color_off[1] : 0; }

// R = B - A X (FP64) -> level-0 B32, X32 and per-column ||R||^2 into scal[8 + c].
template <int NR>
static gmg_status outer_m(gmg_ctx* c, const double* X, cudaStream_t s) {
  Level& L = c->L[0];
  constexpr int Q = NR < 2 ? 1 : NR / 2;
  const int64_t nb = std::min<int64_t>(kRedBlocks, (L.A.nslice * Q + 7) / 8);
  return launch(k_outer_residual_m<NR>, nb, 256, s, L.A.nslice, L.A.ptr, L.A.row0, L.A.nrow, L.A.col, L.A.v64,
                L.diag64, X, (const double*)c->BS, L.B32, L.X32, (const float*)L.dinv32, first_rows(c), c->red,
                c->red_cnt + 3, c->scal + 8);
}

template <int NR>
static gmg_status iteration_m(gmg_ctx* c, cudaStream_t s) {
  Level& L = c->L[0];
  GMG_TRY(vcycle_m<NR>(c, 0, s, first_rows(c) > 0));
  GMG_TRY(launch(k_add_f2d_m, gblk((L.n * NR + 3) / 4), 256, s, L.n * NR, (const float*)L.X32, c->XS));
  return outer_m<NR>(c, c->XS, s);
}

static gmg_status ensure_batched(gmg_ctx* c) {
  if (c->XS) return GMG_OK;
  for (auto& L : c->L) {
    GMG_TRY(c->arena.alloc(&L.X32, (size_t)L.n * kMaxRhs));
    GMG_TRY(c->arena.alloc(&L.B32, (size_t)L.n * kMaxRhs));
    GMG_TRY(c->arena.alloc(&L.R32, (size_t)L.n * kMaxRhs));
  }
  const int64_t n = c->L[0].n;
  GMG_TRY(c->arena.alloc(&c->BS, (size_t)n * kMaxRhs));
  GMG_TRY(c->arena.alloc(&c->RS, (size_t)n * kMaxRhs));
  // per-column partials of the batched residual, and never smaller than the
  // single-vector partials the buffer already serves
  const int64_t need = std::max<int64_t>((int64_t)kRedBlocks * kMaxRhs, c->red_cap);
  double* red2;
  GMG_TRY(c->arena.alloc(&red2, (size_t)need));
  c->red = red2;
  c->red_cap = need;
  // last: it says that all of them are there (a call that ran out of memory on
  // the way leaves it null, and the next one starts again)
  return c->arena.alloc(&c->XS, (size_t)n * kMaxRhs);
}

// The device-side loop of the batched solve for blocks of NR columns: a graph
// whose conditional WHILE node repeats one iteration and its convergence test
// (programmatic launch edges kept where the CUDA driver instantiates them,
// else plain stream order).  Leaves mloops[slot] null when refused.
template <int NR>
static gmg_status build_mloop(gmg_ctx* c) {
  const int slot = nr_index(NR);
  if (!c->g_stream) GMG_CK(cudaStreamCreateWithFlags(&c->g_stream, cudaStreamNonBlocking));
  for (int attempt = 0; attempt < 2 && !c->mloops[slot]; ++attempt) {
    cudaGraph_t g = nullptr;
    GMG_CK(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle h = 0;
    cudaGraphNodeParams np = {};
    cudaError_t e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess) {
      np.type = cudaGraphNodeTypeConditional;
      np.conditional.handle = h;
      np.conditional.type = cudaGraphCondTypeWhile;
      np.conditional.size = 1;
      cudaGraphNode_t node;
      e = cudaGraphAddNode(&node, g, nullptr, nullptr, 0, &np);
    }
    gmg_status st = GMG_OK;
    if (e == cudaSuccess) {
      const uint64_t before = g_launches;
      g_pdl_suspended = attempt == 1;
      e = cudaStreamBeginCaptureToGraph(c->g_stream, np.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                        cudaStreamCaptureModeThreadLocal);
      if (e == cudaSuccess) {
        st = iteration_m<NR>(c, c->g_stream);
        if (st == GMG_OK)
          st = launch(k_batched_check, 1, 32, c->g_stream, c->dloop, c->dhist, (const double*)(c->scal + 8),
                      (const double*)(c->scal + 24), (const double*)(c->scal + 40), h);
        cudaGraph_t body = nullptr;
        e = cudaStreamEndCapture(c->g_stream, &body);
      }
      g_pdl_suspended = false;
      c->mloop_kernels[slot] = g_launches - before;
      g_launches = before;
      if (st == GMG_OK && e == cudaSuccess) e = cudaGraphInstantiate(&c->mloops[slot], g, 0);
    }
    cudaGraphDestroy(g);
    if (st != GMG_OK) return st;
    if (e != cudaSuccess) {
      cudaGetLastError();
      c->mloops[slot] = nullptr;
    }
  }
  if (!c->mloops[slot]) c->mloop_refused[slot] = true;
  return GMG_OK;
}

// Forgets the batched loops (their launch shapes are stale).
static void drop_mloops(gmg_ctx* c) {
  for (int q = 0; q < 5; ++q) {
    if (c->mloops[q]) cudaGraphExecDestroy(c->mloops[q]);
    c->mloops[q] = nullptr;
    c->mloop_refused[q] = false;
  }
}

static bool device_loop_off() {
  static const bool off = [] {
    const char* v = std::getenv("GMG_NO_DEVICE_LOOP");
    return v && v[0] == '1';
  }();
  return off;
}

template <int NR>
static gmg_status solve_m(gmg_ctx* c, int nrhs, const double* B, double* X, double tol, int mem,
                          gmg_solve_info* info, cudaStream_t s) {
  Level& L0 = c->L[0];
  const int64_t n = L0.n;
  const size_t bytes = sizeof(double) * (size_t)(n * nrhs);
  const double* bsrc = B;
  const double* xsrc = X;
  if (mem == GMG_MEM_HOST) {
    GMG_CK(cudaMemcpyAsync(c->RS, B, bytes, cudaMemcpyHostToDevice, s));
    bsrc = c->RS;
  }
  k_gather_m<<<gblk(n * NR), 256, 0, s>>>(n, nrhs, NR, L0.perm, bsrc, c->BS);
  LCK();
  if (mem == GMG_MEM_HOST) {
    GMG_CK(cudaMemcpyAsync(c->RS, X, bytes, cudaMemcpyHostToDevice, s));
    xsrc = c->RS;
  }
  k_gather_m<<<gblk(n * NR), 256, 0, s>>>(n, nrhs, NR, L0.perm, xsrc, c->XS);
  LCK();
  // column norms of B: the outer residual with X = 0 (RS as a zero iterate)
  GMG_CK(cudaMemsetAsync(c->scal, 0, 64 * sizeof(double), s));
  double nb[kMaxRhs];
  bool all_zero = true;
  {
    GMG_CK(cudaMemsetAsync(c->RS, 0, sizeof(double) * (size_t)(n * NR), s));
    GMG_TRY(outer_m<NR>(c, c->RS, s));
    GMG_CK(cudaMemcpyAsync(c->h_scal + 8, c->scal + 8, NR * sizeof(double), cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaStreamSynchronize(s));
    int zmask = 0;
    for (int q = 0; q < nrhs; ++q) {
      nb[q] = std::sqrt(c->h_scal[8 + q]);
      if (nb[q] == 0.0) zmask |= 1 << q;
      else all_zero = false;
    }
    if (zmask) {  // a zero right-hand side has the solution 0
      k_zero_cols<<<gblk(n * NR), 256, 0, s>>>(n, NR, zmask, c->XS);
      LCK();
    }
  }
  auto worst = [&]() {
    double w = 0.0;
    for (int q = 0; q < nrhs; ++q) {
      // a norm that is not finite: so is the quotient (0 only where B's column is zero)
      const double r = nb[q] == 0.0 ? 0.0 : std::sqrt(c->h_scal[8 + q]) / nb[q];
      if (!std::isfinite(r)) return r;
      w = std::max(w, r);
    }
    return w;
  };
  GMG_TRY(outer_m<NR>(c, c->XS, s));
  GMG_CK(cudaMemcpyAsync(c->h_scal + 8, c->scal + 8, NR * sizeof(double), cudaMemcpyDeviceToHost, s));
  GMG_CK(cudaStreamSynchronize(s));
  double rel = worst();
  if (info && info->history && info->history_cap > 0) info->history[0] = rel;
  gmg_status st = GMG_ERR_NOT_CONVERGED;
  int k = 0;
  if (!std::isfinite(rel)) {
    st = GMG_ERR_NONFINITE;
  } else if (all_zero) {
    st = GMG_OK;
  } else {
    const int slot = nr_index(NR);
    const bool loop = c->opt.use_graphs && !device_loop_off();
    if (loop && c->opt.max_iter > 0 && !(rel <= tol) && !c->mloops[slot] && !c->mloop_refused[slot])
      GMG_TRY(build_mloop<NR>(c));
    if (loop && c->opt.max_iter > 0 && c->mloops[slot]) {
      // at least one iteration is made, as in the host-driven loop
      const int it[3] = {0, c->opt.max_iter, nrhs};
      double par[17];
      for (int q = 0; q < 16; ++q) par[q] = q < nrhs ? nb[q] : 0.0;
      par[16] = tol;
      GMG_CK(cudaMemcpyAsync(c->scal + 24, par, sizeof(par), cudaMemcpyHostToDevice, s));
      GMG_CK(cudaMemcpyAsync(c->dloop, it, sizeof(it), cudaMemcpyHostToDevice, s));
      GMG_CK(cudaGraphLaunch(c->mloops[slot], s));
      int* hk = reinterpret_cast<int*>(c->h_scal + 40);
      GMG_CK(cudaMemcpyAsync(hk, c->dloop, sizeof(int), cudaMemcpyDeviceToHost, s));
      GMG_CK(cudaMemcpyAsync(c->h_scal + 8, c->scal + 8, NR * sizeof(double), cudaMemcpyDeviceToHost, s));
      GMG_CK(cudaStreamSynchronize(s));
      k = *hk;
      if (k < 1 || k > c->opt.max_iter) {
        set_error("gmg_solve_batched: iteration counter out of range");
        return GMG_ERR_CUDA;
      }
      g_launches += (uint64_t)k * c->mloop_kernels[slot];
      if (info && info->history && info->history_cap > 1)
        GMG_CK(cudaMemcpy(info->history + 1, c->dhist + 1,
                          sizeof(double) * (size_t)std::min(k, info->history_cap - 1), cudaMemcpyDeviceToHost));
      rel = worst();
      st = !std::isfinite(rel) ? GMG_ERR_NONFINITE : rel <= tol ? GMG_OK : GMG_ERR_NOT_CONVERGED;
    } else
    while (k < c->opt.max_iter) {
      GMG_TRY(iteration_m<NR>(c, s));
      GMG_CK(cudaMemcpyAsync(c->h_scal + 8, c->scal + 8, NR * sizeof(double), cudaMemcpyDeviceToHost, s));
      GMG_CK(cudaStreamSynchronize(s));
      ++k;
      rel = worst();
      if (info && info->history && k < info->history_cap) info->history[k] = rel;
      if (!std::isfinite(rel)) {
        st = GMG_ERR_NONFINITE;
        break;
      }
      if (rel <= tol) {
        st = GMG_OK;
        break;
      }
    }
  }
  double* dst = mem == GMG_MEM_HOST ? c->RS : X;
  k_scatter_m<<<gblk(n * nrhs), 256, 0, s>>>(n, nrhs, NR, L0.perm, c->XS, dst);
  LCK();
  if (mem == GMG_MEM_HOST) {
    GMG_CK(cudaMemcpyAsync(X, c->RS, bytes, cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaStreamSynchronize(s));
  }
  if (info) {
    info->iters = k;
    info->rel_res = rel;
  }
  if (st == GMG_ERR_NOT_CONVERGED) set_error("gmg_solve_batched: max_iter reached");
  if (st == GMG_ERR_NONFINITE) set_error("gmg_solve_batched: non-finite residual");
  return st;
}

}  // namespace gmg

using namespace gmg;

extern "C" gmg_status gmg_solve_batched(gmg_handle h, int nrhs, const double* B, double* X, double tol, int mem,
                                        gmg_solve_info* info, void* stream) {
  gmg::NvtxRange nv("gmg_solve_batched");
  if (!h || !B || !X || nrhs < 1 || nrhs > kMaxRhs || !(tol >= 0.0) ||
      (mem != GMG_MEM_HOST && mem != GMG_MEM_DEVICE)) {
    set_error("gmg_solve_batched: bad handle, vector, nrhs (1..16), tolerance or memory kind");
    return GMG_ERR_INVALID_ARG;
  }
  GMG_CK(cudaSetDevice(h->device));
  GMG_TRY(ensure_batched(h));
  cudaStream_t s = (cudaStream_t)stream;
  GMG_TRY(join_inverse(h, s, true));
  if (nrhs == 1) return solve_m<1>(h, nrhs, B, X, tol, mem, info, s);
  if (nrhs == 2) return solve_m<2>(h, nrhs, B, X, tol, mem, info, s);
  if (nrhs <= 4) return solve_m<4>(h, nrhs, B, X, tol, mem, info, s);
  if (nrhs <= 8) return solve_m<8>(h, nrhs, B, X, tol, mem, info, s);
  return solve_m<16>(h, nrhs, B, X, tol, mem, info, s);
}

namespace gmg {
// One FP32 multi-right-hand-side V-cycle on the finest level, X <- MGI32(X, B):
// caller-numbered FP64 blocks in, rounded to FP32, the cycle, widened back.
template <int NR>
static gmg_status vcycle_step_m(gmg_ctx* c, int nrhs, const double* B, double* X, cudaStream_t s) {
  Level& L0 = c->L[0];
  const int64_t n = L0.n;
  k_gather_m<<<gblk(n * NR), 256, 0, s>>>(n, nrhs, NR, L0.perm, B, c->BS);
  LCK();
  k_gather_m<<<gblk(n * NR), 256, 0, s>>>(n, nrhs, NR, L0.perm, X, c->XS);
  LCK();
  GMG_TRY(launch_d2f(n * NR, c->BS, L0.B32, s));
  GMG_TRY(launch_d2f(n * NR, c->XS, L0.X32, s));
  GMG_TRY(vcycle_m<NR>(c, 0, s, false));
  GMG_TRY(launch_f2d(n * NR, L0.X32, c->XS, s));
  k_scatter_m<<<gblk(n * nrhs), 256, 0, s>>>(n, nrhs, NR, L0.perm, c->XS, X);
  LCK();
  return GMG_OK;
}
}  // namespace gmg

extern "C" gmg_status gmg_vcycle_batched(gmg_handle h, int nrhs, const double* B, double* X, void* stream) {
  if (!h || !B || !X || nrhs < 1 || nrhs > kMaxRhs) {
    set_error("gmg_vcycle_batched: bad handle, block or nrhs (1..16)");
    return GMG_ERR_INVALID_ARG;
  }
  GMG_CK(cudaSetDevice(h->device));
  GMG_TRY(ensure_batched(h));
  cudaStream_t s = (cudaStream_t)stream;
  GMG_TRY(join_inverse(h, s, true));
  if (nrhs == 1) return vcycle_step_m<1>(h, nrhs, B, X, s);
  if (nrhs == 2) return vcycle_step_m<2>(h, nrhs, B, X, s);
  if (nrhs <= 4) return vcycle_step_m<4>(h, nrhs, B, X, s);
  if (nrhs <= 8) return vcycle_step_m<8>(h, nrhs, B, X, s);
  return vcycle_step_m<16>(h, nrhs, B, X, s);
}

namespace gmg {
// Times every smoothed level's multi-right-hand-side sweeps (all colours, four
// sweeps) and residual for NR columns with each warps-per-row split G, as
// captured CUDA graphs (the way a solve runs them), and keeps the fastest G.
template <int NR>
static gmg_status autotune_m(gmg_ctx* c, int* lanes_out, cudaStream_t stream) {
  GMG_CK(cudaStreamSynchronize(stream));
  if (!c->g_stream) GMG_CK(cudaStreamCreateWithFlags(&c->g_stream, cudaStreamNonBlocking));
  cudaStream_t cs = c->g_stream;
  cudaEvent_t e0, e1;
  GMG_CK(cudaEventCreate(&e0));
  GMG_CK(cudaEventCreate(&e1));
  const uint64_t launches_before = g_launches;
  gmg_status st = GMG_OK;
  for (int l = 0; l + 1 < c->nlev && st == GMG_OK; ++l) {
    Level& L = c->L[l];
    if (cudaMemsetAsync(L.X32, 0, sizeof(float) * (size_t)(L.n * NR), cs) != cudaSuccess ||
        cudaMemsetAsync(L.B32, 0, sizeof(float) * (size_t)(L.n * NR), cs) != cudaSuccess) {
      st = GMG_ERR_CUDA;
      break;
    }
    float best_ms = 1e30f;
    int best = m_lanes<NR>(L);
    for (int G : {1, 2, 4, 8}) {
      cudaGraph_t g = nullptr;
      cudaGraphExec_t ge = nullptr;
      if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        st = GMG_ERR_CUDA;
        break;
      }
      for (int sweep = 0; sweep < 4 && st == GMG_OK; ++sweep)
        for (int k = 0; k < L.ncolor && st == GMG_OK; ++k) st = sweep_m<NR>(L, k, cs, G);
      if (st == GMG_OK) st = residual_m<NR>(L, cs, G);
      const cudaError_t ec = cudaStreamEndCapture(cs, &g);
      if (st == GMG_OK && ec == cudaSuccess && cudaGraphInstantiate(&ge, g, 0) == cudaSuccess) {
        float ms = 0.f;
        cudaGraphLaunch(ge, cs);  // warm-up
        cudaEventRecord(e0, cs);
        for (int rep = 0; rep < 3; ++rep) cudaGraphLaunch(ge, cs);
        cudaEventRecord(e1, cs);
        if (cudaEventSynchronize(e1) != cudaSuccess) st = GMG_ERR_CUDA;
        cudaEventElapsedTime(&ms, e0, e1);
        if (st == GMG_OK && ms < best_ms) {
          best_ms = ms;
          best = G;
        }
      } else if (st == GMG_OK) {
        set_error("gmg_autotune_batched: graph capture of the sweeps failed");
        st = GMG_ERR_CUDA;
      }
      if (ge) cudaGraphExecDestroy(ge);
      if (g) cudaGraphDestroy(g);
    }
    if (st == GMG_OK) L.mlanes[nr_index(NR)] = best;
    if (lanes_out) lanes_out[l] = L.mlanes[nr_index(NR)];
  }
  g_launches = launches_before;  // timing launches are not the caller's work
  cudaStreamSynchronize(cs);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  drop_mloops(c);
  return st;
}

static int block_width(int nrhs) { return nrhs <= 1 ? 1 : nrhs <= 2 ? 2 : nrhs <= 4 ? 4 : nrhs <= 8 ? 8 : 16; }

static gmg_status autotune_batched(gmg_ctx* c, int nrhs, int* lanes_out, cudaStream_t s) {
  GMG_CK(cudaSetDevice(c->device));
  GMG_TRY(ensure_batched(c));
  switch (block_width(nrhs)) {
    case 1: return autotune_m<1>(c, lanes_out, s);
    case 2: return autotune_m<2>(c, lanes_out, s);
    case 4: return autotune_m<4>(c, lanes_out, s);
    case 8: return autotune_m<8>(c, lanes_out, s);
    default: return autotune_m<16>(c, lanes_out, s);
  }
}
}  // namespace gmg

extern "C" gmg_status gmg_autotune_batched(gmg_handle h, int nrhs, int* lanes_out, void* stream) {
  if (!h || nrhs < 1 || nrhs > kMaxRhs) {
    set_error("gmg_autotune_batched: bad handle or nrhs (1..16)");
    return GMG_ERR_INVALID_ARG;
  }
  return autotune_batched(h, nrhs, lanes_out, (cudaStream_t)stream);
}

extern "C" gmg_status gmg_set_lanes_batched(gmg_handle h, int nrhs, const int* lanes) {
  if (!h || nrhs < 1 || nrhs > kMaxRhs || !lanes) {
    set_error("gmg_set_lanes_batched: bad handle, nrhs (1..16) or null lanes");
    return GMG_ERR_INVALID_ARG;
  }
  for (int l = 0; l + 1 < h->nlev; ++l)
    if (lanes[l] != 1 && lanes[l] != 2 && lanes[l] != 4 && lanes[l] != 8) {
      set_error("gmg_set_lanes_batched: level " + std::to_string(l) + " split " + std::to_string(lanes[l]) +
                " is not 1, 2, 4 or 8");
      return GMG_ERR_INVALID_ARG;
    }
  const int slot = nr_index(block_width(nrhs));
  for (int l = 0; l + 1 < h->nlev; ++l) h->L[l].mlanes[slot] = lanes[l];
  GMG_CK(cudaSetDevice(h->device));
  drop_mloops(h);
  return GMG_OK;
}

// ------------------------------------------------------------------ many meshes
// A batch of independent systems (meshes of uneven size), each with its own
// hierarchy and nrhs right-hand sides.  The whole solve is ONE graph launch:
// a conditional WHILE node repeats an iteration in which a gate kernel opens
// one conditional IF node per mesh that has not converged yet; the IF bodies
// (each mesh's multi-right-hand-side FP32 V-cycle, FP64 correction and FP64
// residual with column norms) run concurrently, and a check kernel then
// updates every mesh's relative residual, iteration count and done flag and
// decides whether the loop goes on.  The host reads the per-mesh results once
// at the end.  Where the CUDA driver refuses the conditional graph, one graph
// per iteration with every mesh's branch and a host-side test is used instead.

struct gmg_many_ctx {
  std::vector<gmg_handle> h;
  cudaStream_t cap = nullptr;
  std::vector<cudaStream_t> br;
  std::vector<cudaEvent_t> ev;
  cudaGraphExec_t graph[5] = {};  // host-driven form, by NR = 1, 2, 4, 8, 16
  uint64_t graph_kernels[5] = {};
  cudaGraphExec_t loop[5] = {};  // device-side loop, by NR
  uint64_t loop_kernels[5] = {};  // kernel nodes of one loop iteration (all meshes open)
  bool loop_refused[5] = {};
  // device state of the device-side loop
  int* d_state = nullptr;        // [0] iterations done, [1] limit, [2] non-finite seen; then per mesh: done, iters
  double* d_nb = nullptr;        // per mesh kMaxRhs column norms of B (0: column unused or zero)
  double* d_rel = nullptr;       // per mesh worst relative residual
  double* d_tol = nullptr;
  double** d_rr = nullptr;       // per mesh: its squared column norms of R (the handle's scal + 8)
  cudaGraphConditionalHandle* d_if = nullptr;  // per mesh IF handle (for the current NR's loop)
  std::vector<cudaGraphConditionalHandle> h_if[5];
};

namespace gmg {

static int nr_slot(int NR) { return NR == 1 ? 0 : NR == 2 ? 1 : NR == 4 ? 2 : NR == 8 ? 3 : 4; }

// Opens the IF node of every mesh that is not done.
__global__ void k_many_gate(int K, const int* __restrict__ state, const cudaGraphConditionalHandle* __restrict__ hif) {
  for (int k = threadIdx.x; k < K; k += blockDim.x) cudaGraphSetConditional(hif[k], state[3 + 2 * k] ? 0u : 1u);
}

// After an iteration: every mesh that ran gets its worst column's relative
// residual and one more iteration, and is done once that is <= tol (a
// non-finite residual ends the whole loop).  The loop continues while a mesh
// is not done and the iteration limit is not reached.  All NR columns of the
// block are tested: the graph serves every call of its width, and the columns
// that a call does not use have norm 0.  One block.
__global__ void k_many_check(int K, int NR, int* state, const double* __restrict__ nb, double* rel,
                             const double* tol, double* const* rr, cudaGraphConditionalHandle hw) {
  __shared__ int open, bad;
  if (threadIdx.x == 0) {
    open = 0;
    bad = 0;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < K; k += blockDim.x) {
    int* st = state + 3 + 2 * k;
    if (st[0]) continue;
    double w = 0.0;
    bool fin = true;
    for (int q = 0; q < NR; ++q) {
      const double b = nb[k * kMaxRhs + q];
      const double r = b == 0.0 ? 0.0 : sqrt(rr[k][q]) / b;
      if (!isfinite(r)) fin = false;
      w = fmax(w, r);
    }
    st[1] += 1;
    rel[k] = fin ? w : (double)NAN;
    if (!fin) atomicOr(&bad, 1);
    if (fin && w <= *tol) st[0] = 1;
    else atomicOr(&open, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const int it = ++state[0];
    if (bad) state[2] = 1;
    cudaGraphSetConditional(hw, (open && !bad && it < state[1]) ? 1u : 0u);
  }
}

// The host-driven form: one graph per iteration with every mesh's branch.
template <int NR>
static gmg_status many_graph(gmg_many_ctx* m, cudaGraphExec_t* out, uint64_t* kernels) {
  const int K = (int)m->h.size();
  const uint64_t before = g_launches;
  GMG_CK(cudaStreamBeginCapture(m->cap, cudaStreamCaptureModeThreadLocal));
  gmg_status st = GMG_OK;
  cudaError_t e = cudaEventRecord(m->ev[K], m->cap);
  for (int k = 0; k < K && st == GMG_OK && e == cudaSuccess; ++k) {
    e = cudaStreamWaitEvent(m->br[k], m->ev[K], 0);
    if (e == cudaSuccess) st = iteration_m<NR>(m->h[k], m->br[k]);
    if (st == GMG_OK && e == cudaSuccess) e = cudaEventRecord(m->ev[k], m->br[k]);
    if (st == GMG_OK && e == cudaSuccess) e = cudaStreamWaitEvent(m->cap, m->ev[k], 0);
  }
  cudaGraph_t g = nullptr;
  cudaError_t ee = cudaStreamEndCapture(m->cap, &g);
  *kernels = g_launches - before;
  g_launches = before;
  if (st != GMG_OK) {
    if (g) cudaGraphDestroy(g);
    return st;
  }
  GMG_CK(e);
  GMG_CK(ee);
  cudaError_t ei = cudaGraphInstantiate(out, g, 0);
  cudaGraphDestroy(g);
  GMG_CK(ei);
  return GMG_OK;
}

// The device-side loop: WHILE { gate -> IF_k { iteration of mesh k } for all k -> check }.
template <int NR>
static gmg_status many_loop(gmg_many_ctx* m, int slot) {
  const int K = (int)m->h.size();
  int width = NR;
  cudaGraph_t g = nullptr;
  GMG_CK(cudaGraphCreate(&g, 0));
  cudaError_t e = cudaSuccess;
  gmg_status st = GMG_OK;
  const uint64_t before = g_launches;
  cudaGraphConditionalHandle hw = 0;
  cudaGraphNodeParams wp = {};
  cudaGraphNode_t wnode;
  e = cudaGraphConditionalHandleCreate(&hw, g, 1, cudaGraphCondAssignDefault);
  if (e == cudaSuccess) {
    wp.type = cudaGraphNodeTypeConditional;
    wp.conditional.handle = hw;
    wp.conditional.type = cudaGraphCondTypeWhile;
    wp.conditional.size = 1;
    e = cudaGraphAddNode(&wnode, g, nullptr, nullptr, 0, &wp);
  }
  cudaGraph_t body = e == cudaSuccess ? wp.conditional.phGraph_out[0] : nullptr;
  std::vector<cudaGraphConditionalHandle>& hif = m->h_if[slot];
  hif.assign(K, 0);
  std::vector<cudaGraphNode_t> ifn(K);
  cudaGraphNode_t gate = nullptr, check = nullptr;
  // gate kernel node (handles are filled into d_if before every launch of this loop)
  if (e == cudaSuccess) {
    cudaKernelNodeParams kp = {};
    void* args[] = {(void*)&K, (void*)&m->d_state, (void*)&m->d_if};
    kp.func = (void*)k_many_gate;
    kp.gridDim = dim3(1);
    kp.blockDim = dim3(256);
    kp.kernelParams = args;
    e = cudaGraphAddKernelNode(&gate, body, nullptr, 0, &kp);
  }
  for (int k = 0; k < K && e == cudaSuccess && st == GMG_OK; ++k) {
    e = cudaGraphConditionalHandleCreate(&hif[k], body, 0, 0);
    if (e != cudaSuccess) break;
    cudaGraphNodeParams ip = {};
    ip.type = cudaGraphNodeTypeConditional;
    ip.conditional.handle = hif[k];
    ip.conditional.type = cudaGraphCondTypeIf;
    ip.conditional.size = 1;
    e = cudaGraphAddNode(&ifn[k], body, &gate, nullptr, 1, &ip);
    if (e != cudaSuccess) break;
    e = cudaStreamBeginCaptureToGraph(m->br[k], ip.conditional.phGraph_out[0], nullptr, nullptr, 0,
                                      cudaStreamCaptureModeThreadLocal);
    if (e != cudaSuccess) break;
    st = iteration_m<NR>(m->h[k], m->br[k]);
    cudaGraph_t cg = nullptr;
    const cudaError_t ec = cudaStreamEndCapture(m->br[k], &cg);
    if (e == cudaSuccess) e = ec;
  }
  if (e == cudaSuccess && st == GMG_OK) {
    cudaKernelNodeParams kp = {};
    void* args[] = {(void*)&K, (void*)&width, (void*)&m->d_state, (void*)&m->d_nb, (void*)&m->d_rel,
                    (void*)&m->d_tol, (void*)&m->d_rr, (void*)&hw};
    kp.func = (void*)k_many_check;
    kp.gridDim = dim3(1);
    kp.blockDim = dim3(256);
    kp.kernelParams = args;
    e = cudaGraphAddKernelNode(&check, body, ifn.data(), (size_t)K, &kp);
  }
  m->loop_kernels[slot] = g_launches - before + 2;
  g_launches = before;
  if (st == GMG_OK && e == cudaSuccess) e = cudaGraphInstantiate(&m->loop[slot], g, 0);
  cudaGraphDestroy(g);
  if (st != GMG_OK) return st;
  if (e != cudaSuccess) {
    cudaGetLastError();
    m->loop[slot] = nullptr;
    m->loop_refused[slot] = true;
    if (const char* v = std::getenv("GMG_VERBOSE"))
      if (v[0] == '1') std::fprintf(stderr, "gmg: many-mesh device loop refused (%s), host loop\n", cudaGetErrorString(e));
  }
  return GMG_OK;
}

template <int NR>
static gmg_status many_solve(gmg_many_ctx* m, int nrhs, const double* const* B, double* const* X, double tol,
                             int mem, gmg_solve_info* info, cudaStream_t s) {
  const int K = (int)m->h.size();
  std::vector<double> nb((size_t)K * kMaxRhs, 0.0);
  std::vector<double> rel(K, 0.0);
  std::vector<int> iters(K, 0), done(K, 0);
  // right-hand sides and initial guesses into every hierarchy's permuted layout
  for (int k = 0; k < K; ++k) {
    gmg_ctx* c = m->h[k];
    Level& L0 = c->L[0];
    const int64_t n = L0.n;
    const size_t bytes = sizeof(double) * (size_t)(n * nrhs);
    const double* bsrc = B[k];
    if (mem == GMG_MEM_HOST) {
      GMG_CK(cudaMemcpyAsync(c->RS, B[k], bytes, cudaMemcpyHostToDevice, s));
      bsrc = c->RS;
    }
    k_gather_m<<<gblk(n * NR), 256, 0, s>>>(n, nrhs, NR, L0.perm, bsrc, c->BS);
    LCK();
    const double* xsrc = X[k];
    if (mem == GMG_MEM_HOST) {
      GMG_CK(cudaMemcpyAsync(c->RS, X[k], bytes, cudaMemcpyHostToDevice, s));
      xsrc = c->RS;
    }
    k_gather_m<<<gblk(n * NR), 256, 0, s>>>(n, nrhs, NR, L0.perm, xsrc, c->XS);
    LCK();
    // ||B_c||: the outer residual of a zero iterate
    GMG_CK(cudaMemsetAsync(c->RS, 0, sizeof(double) * (size_t)(n * NR), s));
    GMG_TRY(outer_m<NR>(c, c->RS, s));
    GMG_CK(cudaMemcpyAsync(c->h_scal + 8, c->scal + 8, NR * sizeof(double), cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaStreamSynchronize(s));
    int zmask = 0;
    for (int q = 0; q < nrhs; ++q) {
      nb[(size_t)k * kMaxRhs + q] = std::sqrt(c->h_scal[8 + q]);
      if (nb[(size_t)k * kMaxRhs + q] == 0.0) zmask |= 1 << q;
    }
    if (zmask) {
      k_zero_cols<<<gblk(n * NR), 256, 0, s>>>(n, NR, zmask, c->XS);
      LCK();
    }
    GMG_TRY(outer_m<NR>(c, c->XS, s));
  }
  // host-side residuals of every mesh not yet done (a done mesh keeps the
  // residual it converged with)
  auto fetch = [&]() -> gmg_status {
    for (int k = 0; k < K; ++k) {
      gmg_ctx* c = m->h[k];
      GMG_CK(cudaMemcpyAsync(c->h_scal + 8, c->scal + 8, NR * sizeof(double), cudaMemcpyDeviceToHost, s));
    }
    GMG_CK(cudaStreamSynchronize(s));
    for (int k = 0; k < K; ++k) {
      if (done[k]) continue;
      double w = 0.0;
      for (int q = 0; q < nrhs; ++q) {
        const double b = nb[(size_t)k * kMaxRhs + q];
        const double r = b == 0.0 ? 0.0 : std::sqrt(m->h[k]->h_scal[8 + q]) / b;
        w = std::isfinite(r) ? std::max(w, r) : r;
        if (!std::isfinite(r)) break;
      }
      rel[k] = w;
    }
    return GMG_OK;
  };
  GMG_TRY(fetch());
  const int slot = nr_slot(NR);
  int max_iter = 0;
  for (auto* c : m->h) max_iter = std::max(max_iter, c->opt.max_iter);
  gmg_status st = GMG_ERR_NOT_CONVERGED;
  bool bad = false, open = false;
  for (int k = 0; k < K; ++k) {
    if (!std::isfinite(rel[k])) bad = true;
    done[k] = rel[k] <= tol;
    if (!done[k]) open = true;
  }
  if (bad) st = GMG_ERR_NONFINITE;
  else if (!open) st = GMG_OK;
  const bool no_loop = device_loop_off();
  if (st == GMG_ERR_NOT_CONVERGED && max_iter > 0 && !no_loop && !m->loop_refused[slot] && !m->loop[slot])
    for (int attempt = 0; attempt < 2 && !m->loop[slot]; ++attempt) {
      g_pdl_suspended = attempt == 1;  // plain stream order if the driver refuses programmatic edges here
      m->loop_refused[slot] = false;
      const gmg_status sl = many_loop<NR>(m, slot);
      g_pdl_suspended = false;
      GMG_TRY(sl);
    }
  if (st == GMG_ERR_NOT_CONVERGED && max_iter > 0 && m->loop[slot]) {
    // device-side loop: state, norms and the IF handles of this loop, one launch
    std::vector<int> hs(3 + 2 * K, 0);
    hs[1] = max_iter;
    for (int k = 0; k < K; ++k) hs[3 + 2 * k] = done[k];
    GMG_CK(cudaMemcpyAsync(m->d_state, hs.data(), sizeof(int) * hs.size(), cudaMemcpyHostToDevice, s));
    GMG_CK(cudaMemcpyAsync(m->d_nb, nb.data(), sizeof(double) * nb.size(), cudaMemcpyHostToDevice, s));
    GMG_CK(cudaMemcpyAsync(m->d_tol, &tol, sizeof(double), cudaMemcpyHostToDevice, s));
    GMG_CK(cudaMemcpyAsync(m->d_rel, rel.data(), sizeof(double) * K, cudaMemcpyHostToDevice, s));
    GMG_CK(cudaMemcpyAsync(m->d_if, m->h_if[slot].data(), sizeof(cudaGraphConditionalHandle) * K,
                           cudaMemcpyHostToDevice, s));
    GMG_CK(cudaGraphLaunch(m->loop[slot], s));
    GMG_CK(cudaMemcpyAsync(hs.data(), m->d_state, sizeof(int) * hs.size(), cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaMemcpyAsync(rel.data(), m->d_rel, sizeof(double) * K, cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaStreamSynchronize(s));
    uint64_t ran = 0;
    for (int k = 0; k < K; ++k) {
      iters[k] = hs[4 + 2 * k];
      done[k] = hs[3 + 2 * k];
      ran += (uint64_t)iters[k];
    }
    // kernels run: per mesh-iteration its share of the body, plus gate and check per iteration
    g_launches += (uint64_t)hs[0] * 2 + (K > 0 ? ran * ((m->loop_kernels[slot] - 2) / (uint64_t)K) : 0);
    bool all = true;
    for (int k = 0; k < K; ++k) all = all && done[k];
    st = hs[2] ? GMG_ERR_NONFINITE : all ? GMG_OK : GMG_ERR_NOT_CONVERGED;
  } else if (st == GMG_ERR_NOT_CONVERGED) {
    // host-driven form: every mesh iterates until all have converged; a
    // mesh's count is the iteration at which it first met the tolerance
    int it = 0;
    while (st == GMG_ERR_NOT_CONVERGED && it < max_iter) {
      if (!m->graph[slot]) GMG_TRY(many_graph<NR>(m, &m->graph[slot], &m->graph_kernels[slot]));
      GMG_CK(cudaGraphLaunch(m->graph[slot], s));
      g_launches += m->graph_kernels[slot];
      ++it;
      GMG_TRY(fetch());
      bool all = true;
      for (int k = 0; k < K; ++k) {
        if (!std::isfinite(rel[k])) bad = true;
        if (!done[k]) {
          iters[k] = it;
          done[k] = rel[k] <= tol;
        }
        all = all && done[k];
      }
      if (bad) st = GMG_ERR_NONFINITE;
      else if (all) st = GMG_OK;
    }
  }
  for (int k = 0; k < K; ++k) {
    gmg_ctx* c = m->h[k];
    const int64_t n = c->L[0].n;
    double* dst = mem == GMG_MEM_HOST ? c->RS : X[k];
    k_scatter_m<<<gblk(n * nrhs), 256, 0, s>>>(n, nrhs, NR, c->L[0].perm, c->XS, dst);
    LCK();
    if (mem == GMG_MEM_HOST)
      GMG_CK(cudaMemcpyAsync(X[k], c->RS, sizeof(double) * (size_t)(n * nrhs), cudaMemcpyDeviceToHost, s));
    if (info) {
      info[k].iters = iters[k];
      info[k].rel_res = rel[k];
    }
  }
  GMG_CK(cudaStreamSynchronize(s));
  if (st == GMG_ERR_NOT_CONVERGED) set_error("gmg_solve_many: max_iter reached");
  if (st == GMG_ERR_NONFINITE) set_error("gmg_solve_many: non-finite residual");
  return st;
}

}  // namespace gmg

extern "C" gmg_status gmg_destroy_many(gmg_many m) {
  if (!m) return GMG_OK;
  for (auto& g : m->graph)
    if (g) cudaGraphExecDestroy(g);
  for (auto& g : m->loop)
    if (g) cudaGraphExecDestroy(g);
  for (void* p : {(void*)m->d_state, (void*)m->d_nb, (void*)m->d_rel, (void*)m->d_tol, (void*)m->d_rr,
                  (void*)m->d_if})
    if (p) cudaFree(p);
  for (auto e : m->ev)
    if (e) cudaEventDestroy(e);
  for (auto s : m->br)
    if (s) cudaStreamDestroy(s);
  if (m->cap) cudaStreamDestroy(m->cap);
  for (auto h : m->h) gmg_destroy(h);
  delete m;
  return GMG_OK;
}

extern "C" gmg_status gmg_setup_many(gmg_many* out, int nmesh, const gmg_csr* A, const int* n_prolong,
                                     const gmg_prolong* const* P, const gmg_options* opt, void* stream) {
  if (!out || nmesh < 1 || !A || !n_prolong || !P) {
    set_error("gmg_setup_many: null argument or nmesh < 1");
    return GMG_ERR_INVALID_ARG;
  }
  *out = nullptr;
  gmg_many_ctx* m = new gmg_many_ctx();
  for (int k = 0; k < nmesh; ++k) {
    gmg_handle h = nullptr;
    gmg_status st = new_handle(&h, &A[k], n_prolong[k], P[k], nullptr, opt, false, stream);
    if (st == GMG_OK) st = ensure_batched(h);
    if (st != GMG_OK) {
      std::string keep = gmg_last_error();
      if (h) gmg_destroy(h);
      gmg_destroy_many(m);
      set_error("mesh " + std::to_string(k) + ": " + keep);
      return st;
    }
    m->h.push_back(h);
  }
  auto ck = [&](cudaError_t e) {
    if (e != cudaSuccess) set_error(std::string("gmg_setup_many: ") + cudaGetErrorString(e));
    return e == cudaSuccess;
  };
  bool ok = ck(cudaStreamCreateWithFlags(&m->cap, cudaStreamNonBlocking));
  m->br.assign(nmesh, nullptr);
  m->ev.assign(nmesh + 1, nullptr);
  for (int k = 0; ok && k < nmesh; ++k) ok = ck(cudaStreamCreateWithFlags(&m->br[k], cudaStreamNonBlocking));
  for (int k = 0; ok && k <= nmesh; ++k) ok = ck(cudaEventCreateWithFlags(&m->ev[k], cudaEventDisableTiming));
  // device state of the device-side loop
  if (ok) ok = ck(cudaMalloc(&m->d_state, sizeof(int) * (size_t)(3 + 2 * nmesh)));
  if (ok) ok = ck(cudaMalloc(&m->d_nb, sizeof(double) * (size_t)nmesh * kMaxRhs));
  if (ok) ok = ck(cudaMalloc(&m->d_rel, sizeof(double) * (size_t)nmesh));
  if (ok) ok = ck(cudaMalloc(&m->d_tol, sizeof(double)));
  if (ok) ok = ck(cudaMalloc(&m->d_rr, sizeof(double*) * (size_t)nmesh));
  if (ok) ok = ck(cudaMalloc(&m->d_if, sizeof(cudaGraphConditionalHandle) * (size_t)nmesh));
  if (ok) {
    std::vector<double*> rr(nmesh);
    for (int k = 0; k < nmesh; ++k) rr[k] = m->h[k]->scal + 8;
    ok = ck(cudaMemcpy(m->d_rr, rr.data(), sizeof(double*) * (size_t)nmesh, cudaMemcpyHostToDevice)) &&
         uploads_landed() == GMG_OK;
  }
  if (!ok) {
    gmg_destroy_many(m);
    return GMG_ERR_CUDA;
  }
  *out = m;
  return GMG_OK;
}

extern "C" gmg_status gmg_solve_many(gmg_many m, int nrhs, const double* const* B, double* const* X, double tol,
                                     int mem, gmg_solve_info* info, void* stream) {
  gmg::NvtxRange nv("gmg_solve_many");
  if (!m || !B || !X || nrhs < 1 || nrhs > kMaxRhs || !(tol >= 0.0) ||
      (mem != GMG_MEM_HOST && mem != GMG_MEM_DEVICE)) {
    set_error("gmg_solve_many: bad handle, vector list, nrhs (1..16), tolerance or memory kind");
    return GMG_ERR_INVALID_ARG;
  }
  for (size_t k = 0; k < m->h.size(); ++k)
    if (!B[k] || !X[k]) {
      set_error("gmg_solve_many: null vector for mesh " + std::to_string(k));
      return GMG_ERR_INVALID_ARG;
    }
  GMG_CK(cudaSetDevice(m->h[0]->device));
  cudaStream_t s = (cudaStream_t)stream;
  if (nrhs == 1) return many_solve<1>(m, nrhs, B, X, tol, mem, info, s);
  if (nrhs == 2) return many_solve<2>(m, nrhs, B, X, tol, mem, info, s);
  if (nrhs <= 4) return many_solve<4>(m, nrhs, B, X, tol, mem, info, s);
  if (nrhs <= 8) return many_solve<8>(m, nrhs, B, X, tol, mem, info, s);
  return many_solve<16>(m, nrhs, B, X, tol, mem, info, s);
}

extern "C" gmg_status gmg_autotune_many(gmg_many m, int nrhs, void* stream) {
  if (!m || nrhs < 1 || nrhs > kMaxRhs) {
    set_error("gmg_autotune_many: bad batch or nrhs (1..16)");
    return GMG_ERR_INVALID_ARG;
  }
  for (size_t k = 0; k < m->h.size(); ++k) {
    gmg_status st = autotune_batched(m->h[k], nrhs, nullptr, (cudaStream_t)stream);
    if (st != GMG_OK) {
      std::string keep = gmg_last_error();
      set_error("mesh " + std::to_string(k) + ": " + keep);
      return st;
    }
  }
  // the captured iterations hold the old launch shapes
  const int slot = nr_index(block_width(nrhs));
  if (m->loop[slot]) cudaGraphExecDestroy(m->loop[slot]);
  if (m->graph[slot]) cudaGraphExecDestroy(m->graph[slot]);
  m->loop[slot] = nullptr;
  m->graph[slot] = nullptr;
  m->loop_refused[slot] = false;
  return GMG_OK;
}
