// The coarse part of a V-cycle (Alg. 2) on one thread-block cluster.
//
// The smoothed levels l0 .. lambda-1 and the coarsest solve run as ONE launch
// on a cluster of 16 CTAs.  Their colour phases are dependent and small (a
// few hundred rows per CTA), so as grid launches each costs a kernel boundary
// and a dependent L2 round trip (2.0-2.9 us measured) whatever its size; here
// a phase is the row arithmetic from shared memory and a cluster barrier.
//
// Rows of a level are split into contiguous ranges of its locality rank, one
// per CTA, so that most neighbours of a row share its CTA and every range
// holds about 1/16 of each colour.  A CTA keeps x of its own rows and of the
// rows of other CTAs that it reads (its halo: neighbours, and the coarse
// parents of its finer rows), b and 1/a_ii of its own rows, and the entries of
// its rows as slices of 32 lanes with 16-bit local columns.  A row that other
// CTAs read is stored into their halo copies through distributed shared
// memory as it is updated.
//
// What bounds a phase is its chain of dependent shared-memory accesses and
// the barrier (16 CTAs of 512 threads: 660 cycles with remote stores,
// measured alone), not bandwidth.  So everything that does not depend on the
// phase before (slice descriptor, first eight entries per lane, b, 1/a_ii,
// list of halo stores) is loaded into registers between the barrier's arrive
// and its wait; after the wait only the gathers of x, the adds, and the
// stores remain.  Levels with few rows per phase split each row over 2, 4 or
// 8 lanes.
//
// Entries stay in shared memory where they fit; the entries of the largest
// levels stream from L2 by TMA bulk copies, one phase's block per stage,
// issued up to three phases ahead.
//
// Levels with at least kClWide rows per phase and CTA keep one thread per row
// and add each row's terms in the order of the level's sliced ELL, so their
// results are those of the per-colour kernels with one warp per row.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <string>
#include <vector>

#include "gmg_cycle.cuh"

namespace gmg {

namespace {

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClPre = 8;    // entries per lane loaded before the phase's wait
constexpr int kClWide = 64;  // rows per phase and CTA from which a level keeps one thread per row
// Entries per phase and CTA up to which a level runs here: above, a phase is
// bound by the shared-memory gathers of 16 SMs and a grid launch over all SMs
// is as fast.
constexpr int64_t kClPhaseEntries = 12288;

__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cl_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cl_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// v into the same shared-memory location of CTA `rank` of the cluster.
__device__ __forceinline__ void cl_store(float* p, unsigned rank, float v) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(ra), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(double* p, unsigned rank, double v) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}
__device__ __forceinline__ void mbar_init(uint64_t* m, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(m)), "r"(count) : "memory");
}
// One arrival that also expects `bytes` of bulk copies to complete on m.
__device__ __forceinline__ void mbar_expect(uint64_t* m, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(m)), "r"(bytes) : "memory");
}
// Bulk copy (TMA engine) of `bytes` (a multiple of 16, both addresses 16-byte
// aligned) from global to this CTA's shared memory, completing on m.
__device__ __forceinline__ void bulk_copy(void* dst, const void* src, unsigned bytes, uint64_t* m) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(m))
               : "memory");
}
// Waits for the phase of m with the given parity to complete; gives up after
// `polls` polls (sets *err) so that a lost copy cannot hang the GPU.  A
// failing poll suspends the warp for about 3.8 us on GB300 (measured with
// gmg_wait_selftest), so the limit gives up after about one second; a poll
// does not advance while the context is switched out.
constexpr int kWaitPolls = 1 << 18;
__device__ __forceinline__ void mbar_wait(uint64_t* m, unsigned parity, int* err, int polls = kWaitPolls) {
  for (int it = 0; it < polls; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(m)), "r"(parity)
        : "memory");
    if (done) return;
  }
  atomicOr(err, 1);
}

// A list of halo stores packed in one word: first entry of the CTA's store
// list << 4 | number of stores (at most 15 other CTAs).
template <class T>
__device__ __forceinline__ void push(T* base, unsigned list, const uint32_t* dst, T v) {
  const uint32_t* d = dst + (list >> 4);
  for (unsigned q = 0; q < (list & 15u); ++q) cl_store(base + (d[q] & 0xFFFFu), d[q] >> 16, v);
}

// What a lane needs of its row before the values of the previous phase.
template <class T>
struct RowPre {
  int row, w, e;  // local row, entries of this lane, first entry
  bool lead;      // this lane writes the row
  T v[kClPre], d;
  int c[kClPre];
  unsigned list;
};

// The row of `lane` in slice `s` (descriptors in `sl`), its first entries, 1/a_ii and halo stores.
template <class T>
__device__ __forceinline__ void load_row_pre(RowPre<T>& p, const int4* sl, int s, int lane, int tpr, int lg,
                                             const T* val, const uint16_t* col, const T* dinv, const uint32_t* xp) {
  const int4 d = sl[s];
  const int ri = lane >> lg;
  const bool in = ri < (d.x >> 16);
  p.row = (d.x & 0xFFFF) + (in ? ri : 0);
  p.w = in ? d.y : 0;
  p.e = d.z + lane;
  p.lead = in && (lane & (tpr - 1)) == 0;
#pragma unroll
  for (int q = 0; q < kClPre; ++q) {
    p.v[q] = q < p.w ? val[p.e + q * 32] : T(0);
    p.c[q] = q < p.w ? col[p.e + q * 32] : 0;
  }
  p.d = p.lead && dinv ? dinv[p.row] : T(0);
  p.list = p.lead ? xp[p.row] : 0u;
}

// sum of the row's a_ij x_j, terms in entry order per lane, the lanes of a
// split row added pairwise (every lane of the row gets the sum).
template <class T>
__device__ __forceinline__ T row_sum(const RowPre<T>& p, const T* val, const uint16_t* col, const T* x, int tpr) {
  T acc = 0;
  T xv[kClPre];
#pragma unroll
  for (int q = 0; q < kClPre; ++q) xv[q] = x[p.c[q]];
#pragma unroll
  for (int q = 0; q < kClPre; ++q)
    if (q < p.w) acc += p.v[q] * xv[q];
  for (int q0 = kClPre; q0 < p.w; q0 += kClPre) {
    T v[kClPre];
    int c[kClPre];
#pragma unroll
    for (int q = 0; q < kClPre; ++q) {
      v[q] = q0 + q < p.w ? val[p.e + (q0 + q) * 32] : T(0);
      c[q] = q0 + q < p.w ? col[p.e + (q0 + q) * 32] : 0;
    }
#pragma unroll
    for (int q = 0; q < kClPre; ++q) xv[q] = x[c[q]];
#pragma unroll
    for (int q = 0; q < kClPre; ++q)
      if (q0 + q < p.w) acc += v[q] * xv[q];
  }
  for (int o = 1; o < tpr; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  return acc;
}

}  // namespace

// x <- MGI(x, b, l0) of Alg. 2 for the levels of D.  With c0_first the rows
// of colour 0 of level l0 have already had their first update from x = 0.
// All CTAs run the same sequence of cluster barriers.
template <class T>
__global__ void __launch_bounds__(kClThreads, 1)
    k_cluster_cycle(const __grid_constant__ ClusterDesc<T> D, T* xg, const T* bg, int c0_first) {
  extern __shared__ __align__(16) char sm[];
  const int cta = (int)cl_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint64_t* mimg = reinterpret_cast<uint64_t*>(sm + D.o_mbar);
  uint64_t* mst = mimg + kClMaxLevels + 1;
  const int NL = D.nlev;  // smoothed levels; lv[NL] is the coarsest
  if (tid == 0) {
    for (int q = 0; q <= NL; ++q) mbar_init(mimg + q, 1);
    for (int q = 0; q < kClStages; ++q) mbar_init(mst + q, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // every level's set-up tables and resident values, before the wait for the previous kernel
  if (tid == 0)
    for (int t = 0; t <= NL; ++t) {
      const ClusterLevel<T>& L = D.lv[t];
      mbar_expect(mimg + t, (unsigned)(L.img_bytes + L.val_bytes));
      bulk_copy(sm + L.o_img, L.img + (int64_t)cta * L.img_bytes, (unsigned)L.img_bytes, mimg + t);
      if (L.val_bytes)
        bulk_copy(sm + L.o_val, L.vimg + (int64_t)cta * L.val_bytes, (unsigned)L.val_bytes, mimg + t);
    }
  // the coarse iterates start from zero, halo copies included
  for (int t = 1; t <= NL; ++t) {
    T* x = reinterpret_cast<T*>(sm + D.lv[t].o_x);
    for (int i = tid; i < D.lv[t].n_loc_max; i += kClThreads) x[i] = T(0);
  }
  mbar_wait(mimg, 0u, D.err);
  // stream step j's entry block (values, then columns) into stage j % nstage
  // (level l0's table starts with the phase of colour 0, skipped with c0_first)
  const int skip = c0_first && D.lv[0].streamed ? 1 : 0;
  const uint2* steps = reinterpret_cast<const uint2*>(sm + D.lv[0].o_img + D.i_steps) + skip;
  const int NS = D.nstage, S = D.nsteps - skip;
  auto issue = [&](int j) {
    if (tid != kClThreads - 32 || j >= S) return;
    const uint2 st = steps[j];
    char* buf = sm + D.o_buf + (j % NS) * D.stage_bytes;
    uint64_t* m = mst + j % NS;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the stage's earlier reads come first
    mbar_expect(m, st.y * (unsigned)(sizeof(T) + 2));
    if (st.y) {
      bulk_copy(buf, D.s_val + st.x, st.y * (unsigned)sizeof(T), m);
      bulk_copy(buf + D.stage_col, D.s_col + st.x, st.y * 2u, m);
    }
  };
  int j = 0;  // next stream step
  if (NS > 0)
    for (int q = 0; q < NS - 1; ++q) issue(q);
  pdl_wait();  // x and b were written by the previous kernels
  pdl_trigger();
  {
    const ClusterLevel<T>& L = D.lv[0];
    const int* hd = reinterpret_cast<const int*>(sm + L.o_img);
    const int nown = hd[0], nloc = hd[1];
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    T* b = reinterpret_cast<T*>(sm + L.o_b);
    const int32_t* l2g = D.l2g + (int64_t)cta * L.n_loc_max;
    for (int i0 = tid; i0 < nloc; i0 += 4 * kClThreads) {
      int g[4];
      T v[4], w[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) g[k] = i0 + k * kClThreads < nloc ? l2g[i0 + k * kClThreads] : 0;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        v[k] = xg[g[k]];
        w[k] = i0 + k * kClThreads < nown ? bg[g[k]] : T(0);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (i0 + k * kClThreads < nloc) x[i0 + k * kClThreads] = v[k];
        if (i0 + k * kClThreads < nown) b[i0 + k * kClThreads] = w[k];
      }
    }
  }
  cl_arrive();
  bool pending = true;  // a cluster barrier has been arrived at and not waited for

  // Gauss-Seidel phases q0 .. nq-1 of level t, colour q mod C (descending:
  // C-1-(q mod C)); b_ready: b of the level was set before the last barrier
  // that this thread waited for.
  auto sweeps = [&](int t, int q0, int nq, bool descending, bool b_ready) {
    const ClusterLevel<T>& L = D.lv[t];
    char* img = sm + L.o_img;
    const int4* sl = reinterpret_cast<const int4*>(img + L.i_sl);
    const int* csl = reinterpret_cast<const int*>(img + L.i_csl);
    const uint32_t* xp = reinterpret_cast<const uint32_t*>(img + L.i_xp);
    const uint32_t* xd = reinterpret_cast<const uint32_t*>(img + L.i_xd);
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    const T* b = reinterpret_cast<const T*>(sm + L.o_b);
    const T* dinv = reinterpret_cast<const T*>(sm + L.o_val);
    const T* val = reinterpret_cast<const T*>(sm + L.o_val + L.v_val);
    const uint16_t* col = reinterpret_cast<const uint16_t*>(img + L.i_col);
    const int C = L.ncolor, tpr = L.tpr, lg = L.lg_tpr;
    int k = q0 % C;
    for (int q = q0; q < nq; ++q) {
      const int kc = descending ? C - 1 - k : k;
      if (++k == C) k = 0;
      if (L.streamed) {
        const char* buf = sm + D.o_buf + (j % NS) * D.stage_bytes;
        val = reinterpret_cast<const T*>(buf);
        col = reinterpret_cast<const uint16_t*>(buf + D.stage_col);
        mbar_wait(mst + j % NS, (unsigned)(j / NS) & 1u, D.err);
      }
      const int s1 = csl[kc + 1];
      int s = csl[kc] + warp;
      RowPre<T> p;
      const bool any = s < s1;
      T bv = 0;
      if (any) {
        load_row_pre<T>(p, sl, s, lane, tpr, lg, val, col, dinv, xp);
        if (b_ready && p.lead) bv = b[p.row];
      }
      if (pending) cl_wait();
      if (L.streamed) {
        issue(j + NS - 1);  // every warp has finished step j - 1
        ++j;
      }
      if (any) {
        if (!b_ready && p.lead) bv = b[p.row];
        for (;;) {
          const T acc = row_sum<T>(p, val, col, x, tpr);
          if (p.lead) {
            const T xn = (bv - acc) * p.d;
            x[p.row] = xn;
            push<T>(x, p.list, xd, xn);
          }
          s += kClWarps;
          if (s >= s1) break;
          load_row_pre<T>(p, sl, s, lane, tpr, lg, val, col, dinv, xp);
          if (p.lead) bv = b[p.row];
        }
      }
      cl_arrive();
      pending = true;
      b_ready = true;
    }
  };

  T* r = reinterpret_cast<T*>(sm + D.o_r);
  T* bc = reinterpret_cast<T*>(sm + D.o_bc);
  for (int t = 0; t < NL; ++t) {
    const ClusterLevel<T>& L = D.lv[t];
    const ClusterLevel<T>& N = D.lv[t + 1];
    char* img = sm + L.o_img;
    const int* hd = reinterpret_cast<const int*>(img);
    const int C = L.ncolor;
    const bool first_done = t == 0 ? c0_first != 0 : D.nu_pre > 0;
    sweeps(t, first_done ? 1 : 0, D.nu_pre * C, false, false);
    // residual of the own rows, stored into the CTAs that restrict it
    {
      const int4* sl = reinterpret_cast<const int4*>(img + L.i_sl);
      const int* csl = reinterpret_cast<const int*>(img + L.i_csl);
      const uint32_t* rp = reinterpret_cast<const uint32_t*>(img + L.i_rp);
      const uint32_t* rd = reinterpret_cast<const uint32_t*>(img + L.i_rd);
      const T* x = reinterpret_cast<const T*>(sm + L.o_x);
      const T* b = reinterpret_cast<const T*>(sm + L.o_b);
      const T* val = reinterpret_cast<const T*>(sm + L.o_val + L.v_val);
      const uint16_t* col = reinterpret_cast<const uint16_t*>(img + L.i_col);
      const T* dg = L.diag + (int64_t)cta * L.n_own_max;
      RowPre<T> p;
      auto load = [&](int s) { load_row_pre<T>(p, sl, s, lane, L.tpr, L.lg_tpr, val, col, dg, rp); };
      auto rows = [&](int s, int se) {  // slices s, s + kClWarps, ..., the first one loaded
        while (s < se) {
          const T acc = row_sum<T>(p, val, col, x, L.tpr);
          if (p.lead) {
            const T rv = b[p.row] - (acc + p.d * x[p.row]);
            r[p.row] = rv;
            push<T>(r, p.list, rd, rv);
          }
          s += kClWarps;
          if (s < se) load(s);
        }
      };
      if (!L.streamed && warp < hd[2]) load(warp);
      if (pending) cl_wait();
      if (!L.streamed) {
        rows(warp, hd[2]);
      } else {
        for (int k = 0; k < C; ++k) {
          const char* buf = sm + D.o_buf + (j % NS) * D.stage_bytes;
          val = reinterpret_cast<const T*>(buf);
          col = reinterpret_cast<const uint16_t*>(buf + D.stage_col);
          issue(j + NS - 1);
          mbar_wait(mst + j % NS, (unsigned)(j / NS) & 1u, D.err);
          if (csl[k] + warp < csl[k + 1]) load(csl[k] + warp);
          rows(csl[k] + warp, csl[k + 1]);
          ++j;
          __syncthreads();
        }
      }
      cl_arrive();
    }
    // restriction b_{l+1} = P^T r over the own coarse rows; x_{l+1} is zero,
    // but the rows of colour 0 of a smoothed level take their first update
    // (b - 0) / a_ii right away.  The first weights are loaded before the wait.
    {
      const int4* rs = L.r_sl + (int64_t)cta * L.rsl_max;
      const int nrs = hd[3], tpr = L.r_tpr, lg = L.lg_r_tpr;
      mbar_wait(mimg + t + 1, 0u, D.err);
      char* nimg = sm + N.o_img;
      const int nc0 = D.nu_pre > 0 && t + 1 < NL ? reinterpret_cast<const int*>(nimg)[4] : 0;
      const uint32_t* xp = reinterpret_cast<const uint32_t*>(nimg + N.i_xp);
      const uint32_t* xd = reinterpret_cast<const uint32_t*>(nimg + N.i_xd);
      const int* gid = reinterpret_cast<const int*>(nimg + N.i_csl);  // coarsest level: global rows of the own rows
      T* xn = reinterpret_cast<T*>(sm + N.o_x);
      T* bn = reinterpret_cast<T*>(sm + N.o_b);
      const T* dn = reinterpret_cast<const T*>(sm + N.o_val);
      constexpr int kR = 16;
      T wv[kR];
      int ci[kR];
      int w = 0, row = 0, e = 0;
      bool lead = false;
      auto terms = [&](int q0) {
#pragma unroll
        for (int q = 0; q < kR; ++q) {
          wv[q] = q0 + q < w ? L.r_w[e + (q0 + q) * 32] : T(0);
          ci[q] = q0 + q < w ? L.r_col[e + (q0 + q) * 32] : 0;
        }
      };
      auto start = [&](int s) {
        const int4 d = rs[s];
        const int ri = lane >> lg;
        const bool in = ri < (d.x >> 16);
        row = (d.x & 0xFFFF) + ri;
        w = in ? d.y : 0;
        e = d.z + lane;
        lead = in && (lane & (tpr - 1)) == 0;
        terms(0);
      };
      int s = warp;
      if (s < nrs) start(s);
      cl_wait();
      for (; s < nrs;) {
        T acc = 0;
        for (int q0 = 0; q0 < w; q0 += kR) {
          T rv[kR];
#pragma unroll
          for (int q = 0; q < kR; ++q) rv[q] = r[ci[q]];
#pragma unroll
          for (int q = 0; q < kR; ++q)
            if (q0 + q < w) acc += wv[q] * rv[q];
          if (q0 + kR < w) terms(q0 + kR);
        }
        for (int o = 1; o < tpr; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (lead) {
          if (t + 1 < NL) {
            bn[row] = acc;
            if (row < nc0) {
              const T v = (acc - T(0)) * dn[row];
              xn[row] = v;
              push<T>(xn, xp[row], xd, v);
            }
          } else {
            for (int c = 0; c < D.ncta; ++c) cl_store(bc + gid[row], (unsigned)c, acc);
          }
        }
        s += kClWarps;
        if (s < nrs) start(s);
      }
      cl_arrive();
      pending = true;
    }
  }
  // coarsest: x_c = A^-1 b_c, one warp per own row, the first row's
  // coefficients loaded before the wait
  {
    const ClusterLevel<T>& L = D.lv[NL];
    char* img = sm + L.o_img;
    const int nown = reinterpret_cast<const int*>(img)[0];
    const int* gid = reinterpret_cast<const int*>(img + L.i_csl);
    const uint32_t* xp = reinterpret_cast<const uint32_t*>(img + L.i_xp);
    const uint32_t* xd = reinterpret_cast<const uint32_t*>(img + L.i_xd);
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    constexpr int kA = sizeof(T) == 4 ? 24 : 12;
    const int n = D.nc;
    T a[kA];
    auto coefs = [&](int i) {
      const T* ar = D.ainv + (int64_t)gid[i] * n;
#pragma unroll
      for (int q = 0; q < kA; ++q) a[q] = lane + 32 * q < n ? ar[lane + 32 * q] : T(0);
    };
    int i = warp;
    if (i < nown) coefs(i);
    cl_wait();
    while (i < nown) {
      T acc = 0;
#pragma unroll
      for (int q = 0; q < kA; ++q)
        if (lane + 32 * q < n) acc += a[q] * bc[lane + 32 * q];
      const T* ar = D.ainv + (int64_t)gid[i] * n;
      for (int q = lane + 32 * kA; q < n; q += 32) acc += ar[q] * bc[q];
      const int cur = i;
      i += kClWarps;
      if (i < nown) coefs(i);
      for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
      if (lane == 0) {
        x[cur] = acc;
        push<T>(x, xp[cur], xd, acc);
      }
    }
    cl_arrive();
    pending = true;
  }
  // up: prolongation and post-smoothing
  for (int t = NL - 1; t >= 0; --t) {
    const ClusterLevel<T>& L = D.lv[t];
    char* img = sm + L.o_img;
    const int nown = reinterpret_cast<const int*>(img)[0];
    const uint32_t* xp = reinterpret_cast<const uint32_t*>(img + L.i_xp);
    const uint32_t* xd = reinterpret_cast<const uint32_t*>(img + L.i_xd);
    T* x = reinterpret_cast<T*>(sm + L.o_x);
    const T* u = reinterpret_cast<const T*>(sm + D.lv[t + 1].o_x);
    const int64_t p0 = (int64_t)cta * 3 * L.n_own_max;
    constexpr int kP = 4;
    int id[kP][3];
    T w[kP][3];
    auto weights = [&](int i0) {
#pragma unroll
      for (int k = 0; k < kP; ++k) {
        const int i = i0 + k * kClThreads < nown ? i0 + k * kClThreads : 0;
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          id[k][m] = L.p_idx[p0 + m * L.n_own_max + i];
          w[k][m] = L.p_w[p0 + m * L.n_own_max + i];
        }
      }
    };
    weights(tid);
    cl_wait();
    for (int i0 = tid; i0 < nown; i0 += kP * kClThreads) {
      if (i0 != tid) weights(i0);
#pragma unroll
      for (int k = 0; k < kP; ++k) {
        const int i = i0 + k * kClThreads;
        if (i < nown) {
          T v = x[i];
          v += w[k][0] * u[id[k][0]] + w[k][1] * u[id[k][1]] + w[k][2] * u[id[k][2]];
          x[i] = v;
          push<T>(x, xp[i], xd, v);
        }
      }
    }
    cl_arrive();
    pending = true;
    sweeps(t, 0, D.nu_post * L.ncolor, !D.post_forward, true);
  }
  if (pending) cl_wait();
  {
    const ClusterLevel<T>& L = D.lv[0];
    const int nown = reinterpret_cast<const int*>(sm + L.o_img)[0];
    const T* x = reinterpret_cast<const T*>(sm + L.o_x);
    const int32_t* l2g = D.l2g + (int64_t)cta * L.n_loc_max;
    for (int i = tid; i < nown; i += kClThreads) xg[l2g[i]] = x[i];
  }
}

// out[e] of every job: the level's value in slot src[e] >= 0, 0 for -1, or
// vector element -2 - src[e] (1/a_ii or a_ii) below.
template <class T>
struct RefreshJobs {
  int njob = 0;
  struct Job {
    int64_t n;
    const int32_t* src;
    const T *val, *vec;
    T* out;
  } job[3 * kClMaxLevels];
};
template <class T>
__global__ void k_cluster_values(const __grid_constant__ RefreshJobs<T> J) {
  const auto& q = J.job[blockIdx.y];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < q.n; e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s = q.src[e];
    q.out[e] = s >= 0 ? q.val[s] : s == -1 ? T(0) : q.vec[-2 - s];
  }
}

// ------------------------------------------------------------------ host

namespace {

template <class T>
cudaLaunchConfig_t cluster_config(const ClusterDesc<T>& D, cudaLaunchAttribute* at, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(D.ncta);
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = (size_t)D.smem;
  cfg.stream = s;
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = D.ncta;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cfg;
}

// Whether the device can run such a cluster (sets the kernel's attributes).
template <class T>
bool cluster_fits(const ClusterDesc<T>& D) {
  if (cudaFuncSetAttribute(k_cluster_cycle<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(k_cluster_cycle<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) !=
          cudaSuccess) {  // the limit every handle's layout stays within
    cudaGetLastError();
    return false;
  }
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg = cluster_config(D, at, nullptr);
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, k_cluster_cycle<T>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return nclusters >= 1;
}

struct Slice {
  int32_t x, y, z, w;  // local row0 | rows << 16, entries per lane, first entry, 0
};

// One CTA's part of a level.
struct Part {
  std::vector<int32_t> own, halo, rhalo;  // permuted rows
  std::vector<Slice> sl, rsl;
  std::vector<int32_t> csl, blk;  // per colour: first slice, first entry (+ end)
  std::vector<uint16_t> ecol, rcol;
  std::vector<int32_t> esrc;
  std::vector<double> rw;
  std::vector<uint32_t> xp, xd, rp, rd;  // halo stores of x and of the residual
  std::vector<uint16_t> pidx;            // 3 x own
  std::vector<double> pw;
  int own0 = 0;  // own rows of colour 0
};
struct Tab {
  int64_t n = 0;
  int ncolor = 0, tpr = 1, r_tpr = 1;
  bool wide = false;
  std::vector<int32_t> owner, local;
  std::vector<Part> part;
  int n_own = 0, n_loc = 0, n_r = 0, nsl = 0, nrsl = 0, nxd = 0, nrd = 0, blk = 0, ent = 0;  // largest over the CTAs
};

int lanes_per_row(double rows, double len) {
  int t = 1;
  while (t < 8 && rows * (2 * t) <= 32 * kClWarps && len >= 4.0 * t) t *= 2;
  return t;
}

// Slices of `rows` rows per slice from rows [0, n) of given lengths; emit(slice, first row, rows, width).
template <class Len, class Emit>
void cut_slices(int i0, int i1, int per, int tpr, Len len, Emit emit) {
  for (int a = i0; a < i1; a += per) {
    const int nr = std::min(per, i1 - a);
    int w = 0;
    for (int q = 0; q < nr; ++q) w = std::max(w, (len(a + q) + tpr - 1) / tpr);
    emit(a, nr, w);
  }
}

// Lists of the halo stores: for each CTA's halo entry (row, local index) the
// owner stores into it.
void push_lists(const std::vector<int32_t>& owner, const std::vector<int32_t>& local, std::vector<Part>& part,
                bool residual) {
  const int ncta = (int)part.size();
  std::vector<std::vector<uint32_t>> cnt(ncta);
  for (int t = 0; t < ncta; ++t) cnt[t].assign(part[t].own.size() + 1, 0);
  for (int t = 0; t < ncta; ++t)
    for (int32_t r : residual ? part[t].rhalo : part[t].halo) ++cnt[owner[r]][local[r] + 1];
  for (int t = 0; t < ncta; ++t) {
    auto& lp = residual ? part[t].rp : part[t].xp;
    auto& ld = residual ? part[t].rd : part[t].xd;
    lp.resize(part[t].own.size());
    for (size_t i = 0; i < part[t].own.size(); ++i) {
      const uint32_t k = cnt[t][i + 1];
      cnt[t][i + 1] += cnt[t][i];
      lp[i] = (cnt[t][i] << 4) | k;
    }
    ld.resize(cnt[t].back());
  }
  for (int t = 0; t < ncta; ++t) {
    const auto& h = residual ? part[t].rhalo : part[t].halo;
    for (size_t q = 0; q < h.size(); ++q) {
      Part& o = part[owner[h[q]]];
      (residual ? o.rd : o.xd)[cnt[owner[h[q]]][local[h[q]]]++] =
          ((uint32_t)t << 16) | (uint32_t)(part[t].own.size() + q);
    }
  }
}

// The tables of levels l0 .. lambda over ncta CTAs (host); false when a local index does not fit 16 bits.
bool build_tables(gmg_ctx* c, int l0, int ncta, const std::vector<std::vector<int64_t>>& hrp,
                  const std::vector<std::vector<int32_t>>& hcol, const std::vector<std::vector<int32_t>>& perm,
                  const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P, std::vector<Tab>& tab) {
  const int lam = c->nlev - 1, nl = lam - l0;
  tab.assign(nl + 1, Tab());
  for (int t = 0; t <= nl; ++t) {
    const Level& L = c->L[l0 + t];
    Tab& T = tab[t];
    T.n = L.n;
    T.ncolor = t < nl ? L.ncolor : 0;
    T.part.assign(ncta, Part());
    T.owner.resize(L.n);
    T.local.resize(L.n);
    for (int64_t r = 0; r < L.n; ++r) {
      const int o = (int)((int64_t)L.h_key[perm[l0 + t][r]] * ncta / L.n);
      T.owner[r] = o;
      T.local[r] = (int32_t)T.part[o].own.size();
      T.part[o].own.push_back((int32_t)r);  // ascending: colour by colour
      if (L.color_off.size() > 1 && r < L.color_off[1]) T.part[o].own0++;
    }
    const double rows = (double)L.n / (std::max(1, L.ncolor) * (double)ncta);
    T.wide = rows >= kClWide;
    T.tpr = T.wide ? 1 : lanes_per_row(rows, (double)(L.nnz - L.n) / (double)L.n);
  }
  std::vector<int32_t> loc, stamp;
  for (int t = 0; t <= nl; ++t) {
    Tab& T = tab[t];
    const int l = l0 + t;
    const int64_t *rp = hrp[l].data();
    const int32_t *ci = hcol[l].data(), *pm = perm[l].data(), *ip = iperm[l].data();
    loc.assign(T.n, 0);
    stamp.assign(T.n, -1);
    for (int a = 0; a < ncta; ++a) {
      Part& p = T.part[a];
      auto see = [&](int32_t r) {
        if (T.owner[r] != a && stamp[r] != a) {
          stamp[r] = a;
          p.halo.push_back(r);
        }
      };
      if (t < nl)
        for (int32_t r : p.own)
          for (int64_t e = rp[pm[r]]; e < rp[pm[r] + 1]; ++e) see(ip[ci[e]]);
      if (t > 0)
        for (int32_t r : tab[t - 1].part[a].own) {
          const int64_t old = perm[l - 1][r];
          for (int s = 0; s < 3; ++s)
            if (P[l - 1].w[3 * old + s] != 0.0) see(ip[P[l - 1].idx[3 * old + s]]);
        }
      std::sort(p.halo.begin(), p.halo.end());
      if (p.own.size() + p.halo.size() > 65535) return false;
      for (size_t q = 0; q < p.halo.size(); ++q) loc[p.halo[q]] = (int32_t)(p.own.size() + q);
      auto at = [&](int32_t r) { return T.owner[r] == a ? T.local[r] : loc[r]; };
      if (t > 0) {  // prolongation slots of the finer level's own rows
        Part& f = tab[t - 1].part[a];
        const size_t m = f.own.size();
        f.pidx.assign(3 * m, 0);
        f.pw.assign(3 * m, 0.0);
        for (size_t i = 0; i < m; ++i) {
          const int64_t old = perm[l - 1][f.own[i]];
          for (int s = 0; s < 3; ++s)
            if (P[l - 1].w[3 * old + s] != 0.0) {
              f.pidx[s * m + i] = (uint16_t)at(ip[P[l - 1].idx[3 * old + s]]);
              f.pw[s * m + i] = P[l - 1].w[3 * old + s];
            }
        }
      }
      if (t < nl) {  // entries in the order of the level's sliced ELL, tpr lanes per row
        const Level& L = c->L[l];
        const int per = 32 / T.tpr;
        auto len = [&](int i) { return (int)(rp[pm[p.own[i]] + 1] - rp[pm[p.own[i]]] - 1); };
        int i0 = 0;
        for (int k = 0; k < T.ncolor; ++k) {
          p.csl.push_back((int32_t)p.sl.size());
          p.blk.push_back((int32_t)p.ecol.size());
          int i1 = i0;
          while (i1 < (int)p.own.size() && p.own[i1] < L.color_off[k + 1]) ++i1;
          cut_slices(i0, i1, per, T.tpr, len, [&](int r0, int nr, int w) {
            const size_t base = p.ecol.size();
            p.sl.push_back({r0 | (nr << 16), w, (int32_t)base, 0});
            p.ecol.resize(base + 32 * (size_t)w);
            p.esrc.resize(base + 32 * (size_t)w, -1);
            for (int q = 0; q < nr; ++q) {
              const int32_t r = p.own[r0 + q];
              const int64_t old = pm[r];
              const int64_t slice = L.color_slice_off[k] + (r - L.color_off[k]) / kSlice;
              const int64_t slot = L.h_ptr[slice] + (r - L.color_off[k]) % kSlice;
              for (int m = 0; m < T.tpr * w; ++m)  // padding: the row itself, value 0
                p.ecol[base + 32 * (size_t)(m / T.tpr) + q * T.tpr + m % T.tpr] = (uint16_t)(r0 + q);
              int m = 0;
              for (int64_t e = rp[old]; e < rp[old + 1]; ++e) {
                if (ci[e] == old) continue;
                const size_t g = base + 32 * (size_t)(m / T.tpr) + q * T.tpr + m % T.tpr;
                p.ecol[g] = (uint16_t)at(ip[ci[e]]);
                p.esrc[g] = (int32_t)(slot + (int64_t)m * kSlice);
                ++m;
              }
            }
          });
          i0 = i1;
          T.blk = std::max(T.blk, (int)p.ecol.size() - p.blk.back());
        }
        p.csl.push_back((int32_t)p.sl.size());
        p.blk.push_back((int32_t)p.ecol.size());
      }
    }
    push_lists(T.owner, T.local, T.part, false);
  }
  // restriction: the own coarse rows gather the residual (fine rows ascending)
  for (int t = 0; t < nl; ++t) {
    Tab &F = tab[t], &N = tab[t + 1];
    const int l = l0 + t;
    const gmg_prolong& p = P[l];
    std::vector<int64_t> cnt(N.n + 1, 0);
    for (int64_t r = 0; r < F.n; ++r) {
      const int64_t old = perm[l][r];
      for (int s = 0; s < 3; ++s)
        if (p.w[3 * old + s] != 0.0) cnt[iperm[l + 1][p.idx[3 * old + s]] + 1]++;
    }
    for (int64_t J = 0; J < N.n; ++J) cnt[J + 1] += cnt[J];
    std::vector<int32_t> tcol(cnt[N.n]);
    std::vector<double> tw(cnt[N.n]);
    {
      std::vector<int64_t> fill(cnt.begin(), cnt.end() - 1);
      for (int64_t r = 0; r < F.n; ++r) {
        const int64_t old = perm[l][r];
        for (int s = 0; s < 3; ++s)
          if (p.w[3 * old + s] != 0.0) {
            const int64_t q = fill[iperm[l + 1][p.idx[3 * old + s]]]++;
            tcol[q] = (int32_t)r;
            tw[q] = p.w[3 * old + s];
          }
      }
    }
    F.r_tpr = F.wide ? 1 : lanes_per_row((double)N.n / ncta, (double)cnt[N.n] / (double)N.n);
    loc.assign(F.n, 0);
    stamp.assign(F.n, -1);
    for (int a = 0; a < ncta; ++a) {
      Part &f = F.part[a], &n = N.part[a];
      for (int32_t J : n.own)
        for (int64_t q = cnt[J]; q < cnt[J + 1]; ++q)
          if (F.owner[tcol[q]] != a && stamp[tcol[q]] != a) {
            stamp[tcol[q]] = a;
            f.rhalo.push_back(tcol[q]);
          }
      std::sort(f.rhalo.begin(), f.rhalo.end());
      if (f.own.size() + f.rhalo.size() > 65535) return false;
      for (size_t q = 0; q < f.rhalo.size(); ++q) loc[f.rhalo[q]] = (int32_t)(f.own.size() + q);
      auto len = [&](int i) { return (int)(cnt[n.own[i] + 1] - cnt[n.own[i]]); };
      cut_slices(0, (int)n.own.size(), 32 / F.r_tpr, F.r_tpr, len, [&](int r0, int nr, int w) {
        const size_t base = f.rcol.size();
        f.rsl.push_back({r0 | (nr << 16), w, (int32_t)base, 0});
        f.rcol.resize(base + 32 * (size_t)w, 0);
        f.rw.resize(base + 32 * (size_t)w, 0.0);
        for (int q = 0; q < nr; ++q) {
          int m = 0;
          for (int64_t k = cnt[n.own[r0 + q]]; k < cnt[n.own[r0 + q] + 1]; ++k, ++m) {
            const size_t g = base + 32 * (size_t)(m / F.r_tpr) + q * F.r_tpr + m % F.r_tpr;
            f.rcol[g] = (uint16_t)(F.owner[tcol[k]] == a ? F.local[tcol[k]] : loc[tcol[k]]);
            f.rw[g] = tw[k];
          }
        }
      });
    }
    push_lists(F.owner, F.local, F.part, true);
  }
  for (Tab& T : tab)
    for (Part& p : T.part) {
      T.n_own = std::max(T.n_own, (int)p.own.size());
      T.n_loc = std::max(T.n_loc, (int)(p.own.size() + p.halo.size()));
      T.n_r = std::max(T.n_r, (int)(p.own.size() + p.rhalo.size()));
      T.nsl = std::max(T.nsl, (int)p.sl.size());
      T.nrsl = std::max(T.nrsl, (int)p.rsl.size());
      T.nxd = std::max(T.nxd, (int)p.xd.size());
      T.nrd = std::max(T.nrd, (int)p.rd.size());
      T.ent = std::max(T.ent, (int)p.ecol.size());
    }
  return true;
}

// Every index the kernel uses: columns and halo stores in range, each halo
// copy written by its row's owner exactly once, slices covering the rows.
bool check_tables(const std::vector<Tab>& tab) {
  const int nl = (int)tab.size() - 1;
  for (int t = 0; t <= nl; ++t) {
    const Tab& T = tab[t];
    for (int kind = 0; kind < (t < nl ? 2 : 1); ++kind) {
      std::vector<std::vector<int>> written(T.part.size());
      for (size_t a = 0; a < T.part.size(); ++a)
        written[a].assign((kind ? T.part[a].rhalo : T.part[a].halo).size(), 0);
      for (size_t a = 0; a < T.part.size(); ++a) {
        const Part& p = T.part[a];
        const auto &lp = kind ? p.rp : p.xp, &ld = kind ? p.rd : p.xd;
        if (lp.size() != p.own.size()) return false;
        for (size_t i = 0; i < lp.size(); ++i)
          for (uint32_t q = 0; q < (lp[i] & 15u); ++q) {
            if ((lp[i] >> 4) + q >= ld.size()) return false;
            const uint32_t d = ld[(lp[i] >> 4) + q], b = d >> 16, li = d & 0xFFFFu;
            if (b >= T.part.size() || b == a) return false;
            const Part& o = T.part[b];
            const auto& h = kind ? o.rhalo : o.halo;
            if (li < o.own.size() || li - o.own.size() >= h.size() || h[li - o.own.size()] != p.own[i]) return false;
            ++written[b][li - o.own.size()];
          }
      }
      for (auto& w : written)
        for (int k : w)
          if (k != 1) return false;
    }
    for (size_t a = 0; a < T.part.size(); ++a) {
      const Part& p = T.part[a];
      if (t < nl) {
        int covered = 0;
        for (const Slice& s : p.sl) {
          if ((s.x & 0xFFFF) != covered || (s.x >> 16) < 1 || (s.x >> 16) * T.tpr > 32 || s.z < 0 ||
              (size_t)s.z + 32 * (size_t)s.y > p.ecol.size())
            return false;
          covered += s.x >> 16;
        }
        if (covered != (int)p.own.size()) return false;
        for (uint16_t q : p.ecol)
          if (q >= std::max<size_t>(1, p.own.size() + p.halo.size())) return false;
        covered = 0;
        for (const Slice& s : p.rsl) {
          if ((s.x & 0xFFFF) != covered || (s.x >> 16) * T.r_tpr > 32 ||
              (size_t)s.z + 32 * (size_t)s.y > p.rcol.size())
            return false;
          covered += s.x >> 16;
        }
        if (covered != (int)tab[t + 1].part[a].own.size()) return false;
        for (uint16_t q : p.rcol)
          if (q >= std::max<size_t>(1, p.own.size() + p.rhalo.size())) return false;
        const Part& n = tab[t + 1].part[a];
        for (uint16_t q : p.pidx)
          if (q >= std::max<size_t>(1, n.own.size() + n.halo.size())) return false;
      }
    }
  }
  return true;
}

template <class T>
gmg_status upload_vec(Arena& a, const T** d, const std::vector<T>& h) {
  T* p;
  GMG_TRY(a.alloc(&p, std::max<size_t>(h.size(), 1)));
  if (!h.empty()) GMG_CK(cudaMemcpy(p, h.data(), h.size() * sizeof(T), cudaMemcpyHostToDevice));
  *d = p;
  return GMG_OK;
}

int64_t al16(int64_t v) { return (v + 15) & ~(int64_t)15; }

// Shared-memory layout: resident levels' entries in shared memory where
// everything fits, the largest levels' entries streamed where not (three
// stages at least, two as a last resort).  False when nothing fits.
template <class T>
bool lay_out(const std::vector<Tab>& tab, int nu_pre, int nu_post, ClusterDesc<T>& D) {
  const int nl = (int)tab.size() - 1;
  std::vector<char> streamed(nl, 0);
  for (;;) {
    int64_t cur = 0, blk = 0;
    int nsteps = 0;
    for (int t = 0; t < nl; ++t)
      if (streamed[t]) {
        nsteps += (nu_pre + 1 + nu_post) * tab[t].ncolor;  // an upper bound: a skipped first phase has no step
        blk = std::max<int64_t>(blk, tab[t].blk);
      }
    D.stage_col = (int)al16(blk * sizeof(T));
    D.stage_bytes = (int)(D.stage_col + al16(2 * blk));
    D.o_mbar = 0;
    cur = al16(8 * (kClMaxLevels + 1 + kClStages));
    int64_t nr = 1;
    for (int t = 0; t <= nl; ++t) {
      const Tab& A = tab[t];
      ClusterLevel<T>& L = D.lv[t];
      const bool res = t < nl && !streamed[t];
      L.streamed = t < nl && streamed[t];
      L.ncolor = A.ncolor;
      L.tpr = A.tpr;
      L.lg_tpr = A.tpr == 1 ? 0 : A.tpr == 2 ? 1 : A.tpr == 4 ? 2 : 3;
      L.r_tpr = A.r_tpr;
      L.lg_r_tpr = A.r_tpr == 1 ? 0 : A.r_tpr == 2 ? 1 : A.r_tpr == 4 ? 2 : 3;
      L.n_own_max = std::max(1, A.n_own);
      L.n_loc_max = std::max(1, A.n_loc);
      L.rsl_max = std::max(1, A.nrsl);
      // image: header, slices, colours (the coarsest level: global rows), halo stores, resident columns, steps
      int64_t o = 32;
      L.i_sl = (int)o;
      o += 16 * (int64_t)A.nsl;
      L.i_csl = (int)o;
      o = al16(o + 4 * (int64_t)(t < nl ? A.ncolor + 1 : L.n_own_max));
      L.i_xp = (int)o;
      o = al16(o + 4 * (int64_t)L.n_own_max);
      L.i_xd = (int)o;
      o = al16(o + 4 * (int64_t)A.nxd);
      L.i_rp = (int)o;
      if (t < nl) o = al16(o + 4 * (int64_t)L.n_own_max);
      L.i_rd = (int)o;
      if (t < nl) o = al16(o + 4 * (int64_t)A.nrd);
      L.i_col = (int)o;
      if (res) o = al16(o + 2 * (int64_t)A.ent);
      if (t == 0) {
        D.i_steps = (int)o;
        o = al16(o + 8 * (int64_t)nsteps);
      }
      L.img_bytes = (int)o;
      L.v_val = (int)al16((int64_t)sizeof(T) * L.n_own_max);
      L.val_bytes = t < nl ? (int)(L.v_val + (res ? al16((int64_t)sizeof(T) * A.ent) : 0)) : 0;
      L.o_img = (int)cur;
      cur += L.img_bytes;
      L.o_val = (int)cur;
      cur += L.val_bytes;
      L.o_x = (int)cur;
      cur = al16(cur + (int64_t)sizeof(T) * L.n_loc_max);
      L.o_b = (int)cur;
      if (t < nl) cur = al16(cur + (int64_t)sizeof(T) * L.n_own_max);
      if (t < nl) nr = std::max<int64_t>(nr, A.n_r);
      if (cur > 4 * (int64_t)kSmemLimit) return false;
    }
    D.o_r = (int)cur;
    cur = al16(cur + (int64_t)sizeof(T) * nr);
    D.o_bc = (int)cur;
    cur = al16(cur + (int64_t)sizeof(T) * tab[nl].n);
    D.o_buf = (int)cur;
    D.nsteps = nsteps;
    const bool all = std::all_of(streamed.begin(), streamed.end(), [](char v) { return v != 0; });
    const int need = blk == 0 ? 0 : all ? 2 : 3;
    if (cur + (int64_t)need * D.stage_bytes <= kSmemLimit) {
      D.nstage = blk == 0 ? 0 : (int)std::min<int64_t>(kClStages, (kSmemLimit - cur) / D.stage_bytes);
      D.smem = (int)(cur + (int64_t)D.nstage * D.stage_bytes);
      return true;
    }
    int big = -1;  // stream the largest level that does not stream yet
    for (int t = 0; t < nl; ++t)
      if (!streamed[t] && (big < 0 || tab[t].ent > tab[big].ent)) big = t;
    if (big < 0) return false;
    streamed[big] = 1;
  }
}

template <class T>
struct Src;
template <>
struct Src<float> {
  static const float* ainv(gmg_ctx* c) { return c->Ainv32; }
  static ClusterDesc<float>& desc(gmg_ctx* c) { return c->cl32; }
};
template <>
struct Src<double> {
  static const double* ainv(gmg_ctx* c) { return c->Ainv; }
  static ClusterDesc<double>& desc(gmg_ctx* c) { return c->cl64; }
};

// Uploads the tables of `tab` in the layout of D.
template <class T>
gmg_status upload_tables(gmg_ctx* c, const std::vector<Tab>& tab, ClusterDesc<T>& D) {
  Arena& a = c->arena;
  const int nl = (int)tab.size() - 1, ncta = D.ncta;
  // streamed entries of all levels, CTA after CTA
  std::vector<uint16_t> s_col;
  std::vector<int32_t> s_src;
  std::vector<std::vector<uint32_t>> s_off(nl);  // per level and CTA: first entry
  for (int t = 0; t < nl; ++t)
    if (D.lv[t].streamed)
      for (const Part& p : tab[t].part) {
        s_off[t].push_back((uint32_t)s_col.size());
        s_col.insert(s_col.end(), p.ecol.begin(), p.ecol.end());
        s_src.insert(s_src.end(), p.esrc.begin(), p.esrc.end());
        D.lv[t].n_stream += (int64_t)p.ecol.size();
      }
  GMG_TRY(upload_vec(a, &D.s_col, s_col));
  T* sv;
  GMG_TRY(a.alloc(&sv, std::max<size_t>(s_col.size(), 1)));
  D.s_val = sv;
  // the stream steps in the kernel's order; the first phase of level l0 has
  // one (the kernel skips it when colour 0 is done), that of a coarser level,
  // done by the restriction, has none
  std::vector<std::vector<uint32_t>> steps(ncta);
  auto step = [&](int t, int k) {
    for (int q = 0; q < ncta; ++q) {
      const Part& p = tab[t].part[q];
      steps[q].push_back(s_off[t][q] + (uint32_t)p.blk[k]);
      steps[q].push_back((uint32_t)(p.blk[k + 1] - p.blk[k]));
    }
  };
  for (int t = 0; t < nl; ++t) {
    if (!D.lv[t].streamed) continue;
    const int C = tab[t].ncolor;
    for (int q = t > 0 ? 1 : 0; q < D.nu_pre * C; ++q) step(t, q % C);
    for (int k = 0; k < C; ++k) step(t, k);
  }
  for (int t = nl - 1; t >= 0; --t) {
    if (!D.lv[t].streamed) continue;
    const int C = tab[t].ncolor;
    for (int q = 0; q < D.nu_post * C; ++q) step(t, D.post_forward ? q % C : C - 1 - q % C);
  }
  D.nsteps = ncta > 0 ? (int)(steps[0].size() / 2) : 0;
  for (int t = 0; t <= nl; ++t) {
    const Tab& A = tab[t];
    ClusterLevel<T>& L = D.lv[t];
    const bool res = t < nl && !L.streamed;
    std::vector<char> img((size_t)ncta * L.img_bytes, 0);
    const size_t nval = (size_t)L.val_bytes / sizeof(T), v0 = (size_t)L.v_val / sizeof(T);
    std::vector<int32_t> vsrc((size_t)ncta * nval, -1), dsrc((size_t)ncta * L.n_own_max, -1);
    std::vector<Slice> rsl((size_t)ncta * L.rsl_max, Slice{0, 0, 0, 0});
    std::vector<uint16_t> rcol, pidx((size_t)ncta * 3 * L.n_own_max, 0);
    std::vector<T> rw, pw((size_t)ncta * 3 * L.n_own_max, T(0));
    std::vector<int32_t> l2g(t == 0 ? (size_t)ncta * L.n_loc_max : 0, 0);
    for (int q = 0; q < ncta; ++q) {
      const Part& p = A.part[q];
      const size_t m = p.own.size();
      char* base = img.data() + (size_t)q * L.img_bytes;
      auto put = [&](int off, const void* v, size_t bytes) {
        if (bytes) std::memcpy(base + off, v, bytes);
      };
      const int32_t hd[8] = {(int32_t)m, (int32_t)(m + p.halo.size()), (int32_t)p.sl.size(), (int32_t)p.rsl.size(),
                             p.own0,     0,                            0,                    0};
      put(0, hd, sizeof(hd));
      std::vector<Slice> sl = p.sl;
      if (L.streamed)  // entry offsets within the colour's block
        for (int k = 0; k < A.ncolor; ++k)
          for (int s = p.csl[k]; s < p.csl[k + 1]; ++s) sl[s].z -= p.blk[k];
      put(L.i_sl, sl.data(), sl.size() * sizeof(Slice));
      if (t < nl) put(L.i_csl, p.csl.data(), p.csl.size() * 4);
      else put(L.i_csl, p.own.data(), m * 4);
      put(L.i_xp, p.xp.data(), p.xp.size() * 4);
      put(L.i_xd, p.xd.data(), p.xd.size() * 4);
      if (t < nl) {
        put(L.i_rp, p.rp.data(), p.rp.size() * 4);
        put(L.i_rd, p.rd.data(), p.rd.size() * 4);
        if (res) put(L.i_col, p.ecol.data(), p.ecol.size() * 2);
        for (size_t i = 0; i < m; ++i) {
          vsrc[(size_t)q * nval + i] = -2 - p.own[i];
          dsrc[(size_t)q * L.n_own_max + i] = -2 - p.own[i];
          for (int s = 0; s < 3; ++s) {
            pidx[((size_t)q * 3 + s) * L.n_own_max + i] = p.pidx[s * m + i];
            pw[((size_t)q * 3 + s) * L.n_own_max + i] = (T)p.pw[s * m + i];
          }
        }
        if (res)
          for (size_t e = 0; e < p.esrc.size(); ++e) vsrc[(size_t)q * nval + v0 + e] = p.esrc[e];
        for (size_t s = 0; s < p.rsl.size(); ++s) {
          rsl[(size_t)q * L.rsl_max + s] = p.rsl[s];
          rsl[(size_t)q * L.rsl_max + s].z += (int32_t)rcol.size();
        }
        rcol.insert(rcol.end(), p.rcol.begin(), p.rcol.end());
        for (double w : p.rw) rw.push_back((T)w);
      }
      if (t == 0) {
        put(D.i_steps, steps[q].data(), steps[q].size() * 4);
        for (size_t i = 0; i < m; ++i) l2g[(size_t)q * L.n_loc_max + i] = p.own[i];
        for (size_t i = 0; i < p.halo.size(); ++i) l2g[(size_t)q * L.n_loc_max + m + i] = p.halo[i];
      }
    }
    GMG_TRY(upload_vec(a, &L.img, img));
    if (t == 0) GMG_TRY(upload_vec(a, &D.l2g, l2g));
    if (t == nl) continue;
    T *vi, *dg;
    GMG_TRY(a.alloc(&vi, std::max<size_t>(vsrc.size(), 1)));
    GMG_TRY(a.alloc(&dg, dsrc.size()));
    L.vimg = reinterpret_cast<const char*>(vi);
    L.diag = dg;
    const int4* d_rsl;
    {
      std::vector<int4> h(rsl.size());
      for (size_t s = 0; s < rsl.size(); ++s) h[s] = make_int4(rsl[s].x, rsl[s].y, rsl[s].z, rsl[s].w);
      GMG_TRY(upload_vec(a, &d_rsl, h));
    }
    L.r_sl = d_rsl;
    GMG_TRY(upload_vec(a, &L.r_col, rcol));
    GMG_TRY(upload_vec(a, &L.r_w, rw));
    GMG_TRY(upload_vec(a, &L.p_idx, pidx));
    GMG_TRY(upload_vec(a, &L.p_w, pw));
    GMG_TRY(upload_vec(a, &L.vsrc, vsrc));
    GMG_TRY(upload_vec(a, &L.dsrc, dsrc));
    L.nvsrc = (int64_t)vsrc.size();
    L.ndsrc = (int64_t)dsrc.size();
  }
  return upload_vec(a, &D.s_src, s_src);
}

template <class T>
gmg_status build_one(gmg_ctx* c, const std::vector<std::vector<int64_t>>& hrp,
                     const std::vector<std::vector<int32_t>>& hcol, const std::vector<std::vector<int32_t>>& perm,
                     const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P) {
  ClusterDesc<T>& D = Src<T>::desc(c);
  D = ClusterDesc<T>{};
  D.l0 = -1;
  const int lam = c->nlev - 1;
  auto env = [](const char* name) {
    const char* e = std::getenv(name);
    return e && e[0] == '1';
  };
  if (lam < 1 || env("GMG_NO_TAIL")) return GMG_OK;
  const bool small_only = env("GMG_NO_CLUSTER_LEVEL");
  std::vector<int> sizes = {16, 8};
  if (const char* e = std::getenv("GMG_TAIL_CTAS")) sizes = {std::atoi(e)};
  for (int ncta : sizes) {
    if (ncta < 1 || ncta > 16) continue;
    for (int l0 = std::max(0, lam - kClMaxLevels); l0 < lam; ++l0) {
      // a quick lower bound of the shared memory before the tables are built
      int64_t least = 4 * c->L[lam].n;
      bool skip = false;
      for (int l = l0; l < lam; ++l) {
        const Level& L = c->L[l];
        const int64_t rows = L.n / (std::max(1, L.ncolor) * ncta);
        skip = skip || (L.nnz - L.n) / (std::max(1, L.ncolor) * (int64_t)ncta) > kClPhaseEntries ||
               (small_only && rows >= kClWide) || L.A.entries > INT32_MAX;
        least += (L.n / ncta) * (int64_t)(3 * sizeof(T) + 8);
      }
      if (skip || least > kSmemLimit) continue;
      std::vector<Tab> tab;
      if (!build_tables(c, l0, ncta, hrp, hcol, perm, iperm, P, tab)) continue;
      // where the ranks are not local (random order: 11-13 halo stores per
      // row on a kNN cloud) a phase would store nearly every row into every CTA
      bool local = true;
      for (int t = 0; t < lam - l0; ++t) {
        int64_t stores = 0;
        for (const Part& p : tab[t].part) stores += (int64_t)p.xd.size();
        local = local && (!tab[t].wide || stores <= 3 * tab[t].n);
      }
      if (!local) continue;
      ClusterDesc<T> E{};
      E.l0 = l0;
      E.ncta = ncta;
      E.nlev = lam - l0;
      E.nc = (int)c->L[lam].n;
      E.nu_pre = c->opt.nu_pre;
      E.nu_post = c->opt.nu_post;
      E.post_forward = c->opt.post_forward;
      if (!lay_out(tab, E.nu_pre, E.nu_post, E)) continue;
      if (!check_tables(tab)) {
        set_error("internal: cluster tables failed their host check");
        return GMG_ERR_INVALID_ARG;
      }
      if (!cluster_fits(E)) break;  // this cluster size cannot be scheduled: try the next
      E.ainv = Src<T>::ainv(c);
      E.err = c->dstatus + 3;
      GMG_CK(cudaMemset(E.err, 0, sizeof(int)));
      GMG_TRY(upload_tables(c, tab, E));
      for (int t = 0; t < E.nlev; ++t) E.wide[t] = tab[t].wide;
      D = E;
      return GMG_OK;
    }
  }
  return GMG_OK;
}

template <class T>
gmg_status refresh_one(gmg_ctx* c, cudaStream_t s) {
  ClusterDesc<T>& D = Src<T>::desc(c);
  if (D.l0 < 0) return GMG_OK;
  RefreshJobs<T> J;
  int64_t most = 1;
  for (int t = 0; t < D.nlev; ++t) {
    Level& L = c->L[D.l0 + t];
    const ClusterLevel<T>& C = D.lv[t];
    const T* v = Vec<T>::v(L.A);
    J.job[J.njob++] = {C.nvsrc, C.vsrc, v, Vec<T>::dinv(L), reinterpret_cast<T*>(const_cast<char*>(C.vimg))};
    J.job[J.njob++] = {C.ndsrc, C.dsrc, v, Vec<T>::diag(L), const_cast<T*>(C.diag)};
    most = std::max(most, C.nvsrc);
  }
  int64_t off = 0;
  for (int t = 0; t < D.nlev; ++t)
    if (D.lv[t].streamed) {
      const int64_t n = D.lv[t].n_stream;
      J.job[J.njob++] = {n, D.s_src + off, Vec<T>::v(c->L[D.l0 + t].A), nullptr, const_cast<T*>(D.s_val) + off};
      off += n;
      most = std::max(most, n);
    }
  k_cluster_values<T><<<dim3((unsigned)std::min<int64_t>((most + 255) / 256, 304), (unsigned)J.njob), 256, 0, s>>>(J);
  GMG_LAUNCHED();
  return GMG_OK;
}

}  // namespace

gmg_status build_cluster(gmg_ctx* c, const std::vector<std::vector<int64_t>>& hrp,
                         const std::vector<std::vector<int32_t>>& hcol, const std::vector<std::vector<int32_t>>& perm,
                         const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P) {
  GMG_TRY(build_one<float>(c, hrp, hcol, perm, iperm, P));
  // FP64 cycles in a solve: the modes that run them
  c->cl64.l0 = -1;
  if (c->opt.precision == GMG_FP64 || c->opt.precision == GMG_FP64_PCG)
    GMG_TRY(build_one<double>(c, hrp, hcol, perm, iperm, P));
  return GMG_OK;
}

gmg_status refresh_cluster_values(gmg_ctx* c, cudaStream_t s) {
  GMG_TRY(refresh_one<float>(c, s));
  return refresh_one<double>(c, s);
}

template <class T>
gmg_status launch_cluster(gmg_ctx* c, T* x, const T* b, bool c0_first, cudaStream_t s) {
  const ClusterDesc<T>& D = Src<T>::desc(c);
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg = cluster_config(D, at, s);
  cfg.numAttrs = use_pdl() ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_cluster_cycle<T>, D, x, b, c0_first ? 1 : 0);
  if (e != cudaSuccess) {
    set_error(std::string("cluster launch: ") + cudaGetErrorString(e));
    return GMG_ERR_CUDA;
  }
  GMG_LAUNCHED();
  return GMG_OK;
}
template gmg_status launch_cluster<float>(gmg_ctx*, float*, const float*, bool, cudaStream_t);
template gmg_status launch_cluster<double>(gmg_ctx*, double*, const double*, bool, cudaStream_t);

// Self-test of the bounded wait: one warp waits on an mbarrier that nothing
// arrives on, so every poll fails and the wait gives up; elapsed device time
// in *ns.
__global__ void k_wait_selftest(int polls, int* err, unsigned long long* ns) {
  __shared__ uint64_t m;
  if (threadIdx.x == 0) mbar_init(&m, 1);
  __syncthreads();
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  mbar_wait(&m, 0u, err, polls);
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
  if (threadIdx.x == 0) *ns = t1 - t0;
}

// GMG_ERR_TIMEOUT once if a cluster launch gave up waiting for an entry block
// (its results are then not to be trusted); clears the flag.
gmg_status cluster_status(gmg_ctx* c, cudaStream_t s) {
  int* err = c->cl32.l0 >= 0 ? c->cl32.err : c->cl64.l0 >= 0 ? c->cl64.err : nullptr;
  if (!err) return GMG_OK;
  int h = 0;
  GMG_CK(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  GMG_CK(cudaStreamSynchronize(s));
  if (h) {
    GMG_CK(cudaMemsetAsync(err, 0, sizeof(int), s));
    set_error("cluster launch: a wait for streamed matrix entries timed out");
    return GMG_ERR_TIMEOUT;
  }
  return GMG_OK;
}

}  // namespace gmg

// The cluster launch's bounded wait run on a barrier that never completes
// (polls <= 0: the limit the solve kernels use).
extern "C" gmg_status gmg_wait_selftest(int polls, int* timed_out, double* ms, void* stream) {
  using namespace gmg;
  if (!timed_out) {
    set_error("gmg_wait_selftest: null pointer");
    return GMG_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  int* err = nullptr;
  unsigned long long* ns = nullptr;
  GMG_CK(cudaMalloc((void**)&err, sizeof(int)));
  if (cudaMalloc((void**)&ns, sizeof(unsigned long long)) != cudaSuccess) {
    cudaFree(err);
    set_error("gmg_wait_selftest: cudaMalloc failed");
    return GMG_ERR_OOM;
  }
  int h = 0;
  unsigned long long hns = 0;
  cudaError_t e = cudaMemsetAsync(err, 0, sizeof(int), s);
  if (e == cudaSuccess) {
    k_wait_selftest<<<1, 32, 0, s>>>(polls > 0 ? polls : kWaitPolls, err, ns);
    ++g_launches;
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hns, ns, sizeof(hns), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  cudaFree(err);
  cudaFree(ns);
  if (e != cudaSuccess) {
    set_error(std::string("gmg_wait_selftest: ") + cudaGetErrorString(e));
    return GMG_ERR_CUDA;
  }
  *timed_out = h;
  if (ms) *ms = 1e-6 * (double)hns;
  return GMG_OK;
}
