// The coarse part of a V-cycle (Alg. 2) on one thread-block cluster.
//
// The smoothed levels l0 .. lambda-1 and the coarsest solve run as ONE launch
// on a cluster of 16 CTAs.  Their colour phases are dependent and small (a
// few hundred rows per CTA), so as grid launches each costs a kernel boundary
// and a dependent L2 round trip (2.0-2.9 us measured) whatever its size; here
// a phase is the row arithmetic from shared memory and a message to the CTAs
// that read its rows.
//
// Rows of a level are split into contiguous ranges of its locality rank, one
// per CTA, so that most neighbours of a row share its CTA and every range
// holds about 1/16 of each colour.  A CTA keeps x of its own rows and of the
// rows of other CTAs that it reads (its halo: neighbours, and the coarse
// parents of its finer rows), b and 1/a_ii of its own rows, and the entries of
// its rows as slices of 32 lanes.  A row that other CTAs read is stored into
// their halo copies through distributed shared memory as it is updated.
//
// What bounds a phase is its chain of dependent steps, not bandwidth, so the
// chain is kept short:
//  * a phase ends with a message, not a barrier: a halo store is an
//    asynchronous remote store that completes on the receiving CTA's
//    mbarrier, each CTA knows how many bytes a phase brings it, and after its
//    own block barrier it waits for those bytes (375 cycles per phase measured
//    alone, against 660 for remote stores and a cluster barrier, whose release
//    has to wait for the stores);
//  * what does not depend on the phase before (slice descriptor, entries,
//    b, 1/a_ii, list of halo stores) is loaded into registers before the wait;
//  * an entry holds the shared-memory address of its x beside its value, two
//    FP32 entries (one FP64) to a 16-byte load;
//  * levels with few rows per phase split each row over 2, 4 or 8 lanes.
// A cycle's levels then take 0.5-0.6 us per phase against 1.1-1.2 us with a
// cluster barrier per phase and 2.0-2.9 us as grid launches.
//
// Messages and skew.  Every phase a CTA also sends a token to each CTA it
// exchanges halo values with, once it has waited for the previous phase.  A
// CTA can therefore be at most one phase ahead of a partner, so that two
// mbarriers, used in turn, tell the phases apart.  A halo value is only
// overwritten after its reader has used it: the phase that overwrites row s
// of a partner's halo waits for the values of all the partner's rows
// adjacent to s that were updated in earlier phases, each sent after it had
// read s (the pattern is symmetric); and between a residual, restriction,
// prolongation and the sweeps around them no array is read in the phase
// before the one that writes it.  Prolongated values of the colour that the
// post-smoothing updates first are not sent: nobody reads them.
//
// Waits that give up.  Every wait on an mbarrier is bounded, and what follows
// one that gave up stays in range and ends:
//  * the tables are waited for before anything is read from them; a CTA that
//    misses one copies them all by plain loads;
//  * a warp that misses a block of entries leaves its rows from then on, and
//    the thread that issues the blocks issues no more;
//  * a lost message leaves an old value in a halo, nothing else; the thread
//    that arms the phase barriers arms none whose last phase it missed, and the
//    messages of a whole cycle stay within a barrier's byte count, so that a
//    CTA that waits no more may run ahead;
//  * every CTA reaches both cluster barriers, since its waits end; before the
//    second it waits, bounded, for its own copies in flight, and after it a CTA
//    that missed something stays a while for messages on their way to it.
// No CTA leaves the phases early: a way out of them, or a function call, cost
// 4 to 7 % of every solve (the compiler then takes the phase loops for
// divergent).  The error word makes later launches wait no more, and the
// solve that reads it report GMG_ERR_TIMEOUT.
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
#include <atomic>
#include <condition_variable>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <functional>
#include <memory>
#include <mutex>
#include <string>
#include <system_error>
#include <thread>
#include <type_traits>
#include <vector>

#include "gmg_cycle.cuh"

namespace gmg {

namespace {

constexpr int kClThreads = 256;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClSlack = 2048;  // shared memory past the last entry unit
// Rows per phase and CTA from which a level keeps one thread per row, with the
// sums of the per-colour kernels (32, 64 and 128 measure alike, within 0.5 %, on
// spheres, tori, the bi-Laplacian and the book: the line is drawn for the bits
// of the large levels, not for speed).
constexpr int kClWide = 64;
// Entries per phase and CTA up to which a level is considered: two stages of
// more would fill the shared memory (FP32: 96 KB each of 227), and the tables
// of levels that cannot fit are not built.
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
__device__ __forceinline__ uint32_t cl_map(uint32_t a, unsigned rank) {
  uint32_t ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(rank));
  return ra;
}
// v to the (cluster) address a, its bytes completing on the mbarrier at m of the same CTA.
__device__ __forceinline__ void cl_send(uint32_t a, uint32_t m, float v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(a),
               "r"(__float_as_uint(v)), "r"(m)
               : "memory");
}
__device__ __forceinline__ void cl_send(uint32_t a, uint32_t m, double v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(a),
               "l"(__double_as_longlong(v)), "r"(m)
               : "memory");
}
__device__ __forceinline__ void mbar_init(uint32_t m, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(m), "r"(count) : "memory");
}
// One arrival that also expects `bytes` of copies or messages to complete on m.
__device__ __forceinline__ void mbar_expect(uint32_t m, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(m), "r"(bytes) : "memory");
}
// Bulk copy (TMA engine) of `bytes` (a multiple of 16, both addresses 16-byte
// aligned) from global to this CTA's shared memory, completing on m.
__device__ __forceinline__ void bulk_copy(uint32_t dst, const void* src, unsigned bytes, uint32_t m) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(m)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t m, unsigned parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(m), "r"(parity)
      : "memory");
  return done != 0;
}
// Waits for the phase of m with the given parity to complete; gives up after
// `polls` polls (sets *err, and polls to 0: the thread waits no more) so that
// a lost copy or message cannot hang the GPU.  A failing poll suspends the
// warp for about 3.8 us on GB300 (measured with gmg_wait_selftest), so the
// limit gives up after about one second; a poll does not advance while the
// context is switched out.
constexpr int kWaitPolls = 1 << 18;
__device__ __forceinline__ void mbar_wait(uint32_t m, unsigned parity, int* err, int& polls) {
#pragma unroll 1
  for (int it = 0; it < polls; ++it)
    if (mbar_try(m, parity)) return;
  atomicOr(err, 1);
  polls = 0;
}

// Shared-memory accesses by 32-bit address, kept in program order with the
// waits (the sweeps are written with them: a phase is some eighty dependent
// instructions per warp, and address arithmetic on generic pointers doubled
// that).
__device__ __forceinline__ uint4 lds4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void lds_pair(uint32_t a, float& x, float& y) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "r"(a));
}
__device__ __forceinline__ void lds_pair(uint32_t a, double& x, double& y) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(x), "=d"(y) : "r"(a));
}
__device__ __forceinline__ void lds1(uint32_t a, float& x) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(x) : "r"(a)); }
__device__ __forceinline__ void lds1(uint32_t a, double& x) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(x) : "r"(a)); }
__device__ __forceinline__ void lds1(uint32_t a, int& x) { asm volatile("ld.shared.s32 %0, [%1];" : "=r"(x) : "r"(a)); }
__device__ __forceinline__ void sts(uint32_t a, float v) { asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory"); }
__device__ __forceinline__ void sts(uint32_t a, double v) { asm volatile("st.shared.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory"); }

// The same under a predicate (no branch).
__device__ __forceinline__ void sts_if(bool p, uint32_t a, float v) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.f32 [%0], %1;\n\t}" ::"r"(a), "f"(v),
               "r"((unsigned)p)
               : "memory");
}
__device__ __forceinline__ void sts_if(bool p, uint32_t a, double v) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.shared.f64 [%0], %1;\n\t}" ::"r"(a), "d"(v),
               "r"((unsigned)p)
               : "memory");
}
__device__ __forceinline__ void cl_send_if(bool p, uint32_t a, uint32_t m, float v) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
      "@p st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];\n\t}" ::"r"(a),
      "r"(__float_as_uint(v)), "r"(m), "r"((unsigned)p)
      : "memory");
}
__device__ __forceinline__ void cl_send_if(bool p, uint32_t a, uint32_t m, double v) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t"
      "@p st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];\n\t}" ::"r"(a),
      "l"(__double_as_longlong(v)), "r"(m), "r"((unsigned)p)
      : "memory");
}

// A halo store in one word: CTA << 28 | local index there << 14 | local index
// here (16,384 local rows of 16 or more bytes would not fit a CTA).
constexpr int kClMaxLocal = 1 << 14;
__device__ __forceinline__ unsigned store_cta(int d) { return (unsigned)d >> 28; }
__device__ __forceinline__ uint32_t store_there(int d) { return ((uint32_t)d >> 14) & 16383u; }
__device__ __forceinline__ uint32_t store_row(int d) { return (uint32_t)d & 16383u; }

// Halo stores e = e0 + k * step of a list, e < e1, of the array at `base` (the
// same address in every CTA), messages to m.
template <class T>
__device__ __forceinline__ void push_list(uint32_t list, int e0, int e1, int step, uint32_t base, uint32_t m) {
#pragma unroll 1
  for (int e = e0; e < e1; e += step) {
    int d;
    lds1(list + 4u * (uint32_t)e, d);
    const uint32_t a = base + store_there(d) * (uint32_t)sizeof(T), to = cl_map(a, store_cta(d));
    T v;
    lds1(base + store_row(d) * (uint32_t)sizeof(T), v);
    cl_send(to, to + (m - a), v);  // the barrier lies in the same CTA's window
  }
}

// acc += the terms of one entry unit: two FP32 entries (value, byte offset of
// x) or one FP64 entry (value, offset, unused).
__device__ __forceinline__ void unit_gather(const uint4& u, uint32_t sm0, float (&x)[2]) {
  lds1(sm0 + u.y, x[0]);
  lds1(sm0 + u.w, x[1]);
}
__device__ __forceinline__ void unit_add(const uint4& u, const float (&x)[2], float& acc) {
  acc += __uint_as_float(u.x) * x[0];
  acc += __uint_as_float(u.z) * x[1];
}
__device__ __forceinline__ void unit_gather(const uint4& u, uint32_t sm0, double (&x)[1]) { lds1(sm0 + u.z, x[0]); }
__device__ __forceinline__ void unit_add(const uint4& u, const double (&x)[1], double& acc) {
  acc += __hiloint2double((int)u.y, (int)u.x) * x[0];
}
template <class T>
constexpr int kPerUnit = sizeof(T) == 4 ? 2 : 1;

// The sum of a row: its w2 pairs of units in order, the first two pairs in u,
// the rest from address ea on (a lane's units lie 512 bytes apart); then the
// lanes of a split row are added pairwise (every lane of the row gets the
// sum).  w2 is the same for the warp.  The next pair is loaded while the
// current one is added, without a test (up to two units past the row's, which
// the layout keeps inside the shared memory).
__device__ __forceinline__ void load_units(uint4 (&u)[4], uint32_t ea) {
#pragma unroll
  for (int q = 0; q < 4; ++q) u[q] = lds4(ea + 512u * q);
}
template <class T>
__device__ __forceinline__ T row_sum(uint4 (&u)[4], uint32_t ea, int w2, uint32_t sm0, int tpr) {
  T acc = 0;
#pragma unroll 1
  for (;;) {
    T xa[kPerUnit<T>], xb[kPerUnit<T>];
    unit_gather(u[0], sm0, xa);
    unit_gather(u[1], sm0, xb);
    unit_add(u[0], xa, acc);
    unit_add(u[1], xb, acc);
    if (--w2 <= 0) break;
    u[0] = u[2];
    u[1] = u[3];
    ea += 1024u;
    u[2] = lds4(ea + 1024u);
    u[3] = lds4(ea + 1536u);
  }
  if (tpr > 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (tpr > 2) {
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      if (tpr > 4) acc += __shfl_xor_sync(0xffffffffu, acc, 4);
    }
  }
  return acc;
}

// Asks L2 for `bytes` from p (a kernel's later reads of set-up data, which the
// finest level's sweeps may have pushed out).
__device__ __forceinline__ void l2_prefetch(const void* p, int64_t bytes, int tid, int nt = kClThreads) {
  const char* c = reinterpret_cast<const char*>(p);
#pragma unroll 1
  for (int64_t o = (int64_t)tid * 128; o < bytes; o += (int64_t)nt * 128)
    asm volatile("prefetch.global.L2 [%0];" ::"l"(c + o));
}

// Stays 0.1 ms for messages that may be on their way to a CTA that missed some.
__device__ __forceinline__ void linger() {
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
#pragma unroll 1
  for (int it = 0; it < 1024; ++it) {
    __nanosleep(500);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
    if (t1 - t0 > 100000) break;
  }
}

}  // namespace

// x <- MGI(x, b, l0) of Alg. 2 for the levels of D.  With c0_first the rows
// of colour 0 of level l0 have already had their first update from x = 0.
// All CTAs run the same sequence of phases.  A: type of the coarsest solve's
// coefficients and sums (a kernel of its own for each: with both in one the
// registers of the phases ran out, 6 us a cycle).
template <class T, class A>
__global__ void __launch_bounds__(kClThreads, 1)
    k_cluster_cycle(const __grid_constant__ ClusterDesc<T> D, T* xg, const T* bg, int c0_first) {
  extern __shared__ __align__(16) char smem[];
  // the base of the shared memory in a register that the compiler keeps: in a
  // cluster launch it forms the address from special registers wherever the
  // array is named, some ten times a phase
  uint32_t sm0;
  asm volatile("mov.u32 %0, %1;" : "=r"(sm0) : "r"(smem_addr(smem)));
  char* sm;
  asm volatile("cvta.shared.u64 %0, %1;" : "=l"(sm) : "l"((uint64_t)sm0));
  const int cta = (int)cl_rank();
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t mimg = sm0 + (uint32_t)D.o_mbar, mst = mimg + 8u * (kClMaxLevels + 1);
  const uint32_t mph = mst + 8u * kClStages, mbc = mph + 16u;  // two phase barriers, the coarsest right-hand side's
  const int NL = D.nlev;  // smoothed levels; lv[NL] is the coarsest
  const A* ainv;
  if constexpr (std::is_same<A, T>::value) ainv = D.ainv;
  else ainv = D.ainv64;
  // after a wait that gave up in an earlier launch nothing is worth waiting for
  int polls = *reinterpret_cast<volatile int*>(D.err) ? 0 : D.polls;
  if (tid == 0) {
#pragma unroll 1
    for (int q = 0; q <= NL; ++q) mbar_init(mimg + 8u * q, 1);
#pragma unroll 1
    for (int q = 0; q < kClStages; ++q) mbar_init(mst + 8u * q, 1);
#pragma unroll 1
    for (int q = 0; q < 2; ++q) mbar_init(mph + 8u * q, 1);
    mbar_init(mbc, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  // every level's set-up tables and resident values, before the wait for the previous kernel
  if (tid == 0)
#pragma unroll 1
    for (int t = 0; t <= NL; ++t) {
      const ClusterLevel<T>& L = D.lv[t];
      mbar_expect(mimg + 8u * t, (unsigned)(L.img_bytes + L.val_bytes));
      bulk_copy(sm0 + (uint32_t)L.o_img, L.img + (int64_t)cta * L.img_bytes, (unsigned)L.img_bytes, mimg + 8u * t);
      if (L.val_bytes)
        bulk_copy(sm0 + (uint32_t)L.o_val, L.vimg + (int64_t)cta * L.val_bytes, (unsigned)L.val_bytes,
                  mimg + 8u * t);
    }
  // the transfers' weights are read once, late: into L2 now
#pragma unroll 1
  for (int t = 0; t < NL; ++t) {
    const ClusterLevel<T>& L = D.lv[t];
    l2_prefetch(L.p_idx + (int64_t)cta * 3 * L.n_own_max, 6 * (int64_t)L.n_own_max, tid);
    l2_prefetch(L.p_w + (int64_t)cta * 3 * L.n_own_max, 3 * (int64_t)sizeof(T) * L.n_own_max, tid);
    l2_prefetch(L.r_col + (int64_t)cta * L.r_max, 2 * (int64_t)L.r_max, tid);
    l2_prefetch(L.r_w + (int64_t)cta * L.r_max, (int64_t)sizeof(T) * L.r_max, tid);
  }
  // the coarse iterates start from zero, halo copies included
#pragma unroll 1
  for (int t = 1; t <= NL; ++t) {
    T* x = reinterpret_cast<T*>(sm + D.lv[t].o_x);
#pragma unroll 1
    for (int i = tid; i < D.lv[t].n_loc_max; i += kClThreads) x[i] = T(0);
  }
#pragma unroll 1
  for (int q = 0; q <= NL; ++q) mbar_wait(mimg + 8u * q, 0u, D.err, polls);
  if (__syncthreads_or(polls == 0)) {  // by plain loads then: what follows indexes with them
#pragma unroll 1
    for (int t = 0; t <= NL; ++t) {
      const ClusterLevel<T>& L = D.lv[t];
      const int* img = reinterpret_cast<const int*>(L.img + (int64_t)cta * L.img_bytes);
      const int* val = reinterpret_cast<const int*>(L.vimg + (int64_t)cta * L.val_bytes);
#pragma unroll 1
      for (int i = tid; i < L.img_bytes / 4; i += kClThreads) reinterpret_cast<int*>(sm + L.o_img)[i] = img[i];
#pragma unroll 1
      for (int i = tid; i < L.val_bytes / 4; i += kClThreads) reinterpret_cast<int*>(sm + L.o_val)[i] = val[i];
    }
    __syncthreads();
  }
  // stream step j's entry block into stage j % nstage (level l0's table
  // starts with the phase of colour 0, skipped with c0_first)
  const int skip = c0_first && D.lv[0].streamed ? 1 : 0;
  const uint2* steps = reinterpret_cast<const uint2*>(sm + D.lv[0].o_img + D.i_steps) + skip;
  const int NS = D.nstage, S = D.nsteps - skip;
  int j = 0, jst = 0;     // next stream step to use, its stage
  unsigned jpar = 0;      // and that stage's parity
  int ji = 0, jist = 0;   // next step to issue, its stage
  int issued = 0;         // steps issued (the issuing thread's)
  auto issue = [&]() {
    if (ji < S && tid == kClThreads - 32 && polls > 0) {
      issued = ji + 1;
      const uint2 st = steps[ji];
      const uint32_t m = mst + 8u * (uint32_t)jist;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the stage's earlier reads come first
      mbar_expect(m, st.y * 16u);
      if (st.y) bulk_copy(sm0 + (uint32_t)(D.o_buf + jist * D.stage_bytes), D.s_ent + st.x, st.y * 16u, m);
    }
    ++ji;
    if (++jist == NS) jist = 0;
  };
  auto stage_used = [&]() {
    ++j;
    if (++jst == NS) {
      jst = 0;
      jpar ^= 1u;
    }
  };
#pragma unroll 1
  for (int q = 0; q + 1 < NS; ++q) issue();
  const int* partners = reinterpret_cast<const int*>(sm + D.lv[0].o_img + D.i_partners);
  const int npart = reinterpret_cast<const int*>(sm + D.lv[0].o_img)[7];
  // global rows of the CTA's rows of level l0 (first ones), before the wait
  const int n0own = reinterpret_cast<const int*>(sm + D.lv[0].o_img)[0];
  const int n0loc = reinterpret_cast<const int*>(sm + D.lv[0].o_img)[1];
  const int32_t* l2g = D.l2g + (int64_t)cta * D.lv[0].n_loc_max;
  constexpr int kX = 8;
  int g[kX];
#pragma unroll
  for (int k = 0; k < kX; ++k) g[k] = tid + k * kClThreads < n0loc ? l2g[tid + k * kClThreads] : 0;
#pragma unroll 1
  for (int i = warp; i < reinterpret_cast<const int*>(sm + D.lv[NL].o_img)[0]; i += kClWarps) {
    const int64_t row = reinterpret_cast<const int*>(sm + D.lv[NL].o_img + D.lv[NL].i_cr)[i];
    l2_prefetch(ainv + row * D.nc, (int64_t)sizeof(A) * D.nc, lane, 32);
  }
  pdl_wait();  // x and b were written by the previous kernels
  pdl_trigger();
  {
    const ClusterLevel<T>& L = D.lv[0];
    const uint32_t a_x = sm0 + (uint32_t)L.o_x, a_bd = sm0 + (uint32_t)L.o_val;
#pragma unroll 1
    for (int i0 = tid; i0 < n0loc; i0 += kX * kClThreads) {
      if (i0 != tid)
#pragma unroll
        for (int k = 0; k < kX; ++k) g[k] = i0 + k * kClThreads < n0loc ? l2g[i0 + k * kClThreads] : 0;
      T v[kX], w[kX];
#pragma unroll
      for (int k = 0; k < kX; ++k) {
        v[k] = xg[g[k]];
        w[k] = i0 + k * kClThreads < n0own ? bg[g[k]] : T(0);
      }
#pragma unroll
      for (int k = 0; k < kX; ++k) {
        const uint32_t o = (uint32_t)sizeof(T) * (uint32_t)(i0 + k * kClThreads);
        if (i0 + k * kClThreads < n0loc) sts(a_x + o, v[k]);
        if (i0 + k * kClThreads < n0own) sts(a_bd + 2u * o, w[k]);
      }
    }
  }
  if (tid == 0)  // what the other CTAs send of the coarsest right-hand side
    mbar_expect(mbc, (unsigned)((D.nc - reinterpret_cast<const int*>(sm + D.lv[0].o_img)[8]) * (int)sizeof(T)));
  cl_arrive();  // every CTA's barriers and copies are set before any message
  cl_wait();

  // Phase p: begin() waits for phase p - 1 (this CTA's threads, then the
  // messages to it; before phase 0 the wait is for the phase before a fresh
  // barrier's first, which counts as complete) and sends this phase's tokens;
  // end(bytes), called by every thread when its messages are on their way,
  // sets the halo bytes that the phase brings.
  int ph = 0;
  const bool sends_token = warp == kClWarps - 1 && lane < npart;
  uint32_t tok_a = 0, tok_m = 0;
  if (sends_token) {
    tok_a = cl_map(sm0 + (uint32_t)D.o_tok + 4u * (uint32_t)cta, (unsigned)partners[lane]);
    tok_m = cl_map(mph, (unsigned)partners[lane]);
  }
  auto mcur = [&]() { return mph + 8u * (uint32_t)(ph & 1); };
  auto begin = [&]() {
    __syncthreads();
    mbar_wait(mph + 8u * (uint32_t)((ph - 1) & 1), (unsigned)((ph - 1) >> 1) & 1u, D.err, polls);
    cl_send_if(sends_token, tok_a, tok_m + 8u * (uint32_t)(ph & 1), 0.f);
  };
  auto end = [&](int bytes) {
    if (tid == 0 && polls > 0) mbar_expect(mcur(), (unsigned)(bytes + 4 * npart));
    ++ph;
  };

  // Gauss-Seidel phases q0 .. nq-1 of level t, colour q mod C (descending:
  // C-1-(q mod C)); b_ready: b of the level was set before the last phase
  // that this thread waited for.  A warp takes slices warp, warp + kClWarps,
  // ... of the colour, a lane a row or a part of it.  The colour's record
  // (first slice, slices, halo bytes) and the first slice's descriptor are
  // loaded a phase ahead, the slice's entries, b, 1/a_ii and halo stores
  // before the wait.
  auto sweeps = [&](int t, int q0, int nq, bool descending, bool b_ready) {
    const ClusterLevel<T>& L = D.lv[t];
    const int C = L.ncolor, tpr = L.tpr, lg = L.lg_tpr, ri = lane >> lg;
    const bool first_part = (lane & (tpr - 1)) == 0, streamed = L.streamed;
    const uint32_t a_img = sm0 + (uint32_t)L.o_img, a_x = sm0 + (uint32_t)L.o_x, a_bd = sm0 + (uint32_t)L.o_val;
    const uint32_t a_cr = a_img + (uint32_t)L.i_cr, a_xd = a_img + (uint32_t)L.i_xd;
    const uint32_t a_sl = a_img + (uint32_t)L.i_sl + 16u * (uint32_t)warp;
    uint32_t a_ent = a_bd + (uint32_t)L.v_ent + 16u * (uint32_t)lane;
    if (q0 >= nq) return;
    int k = q0 % C;
    uint4 cr = lds4(a_cr + 16u * (uint32_t)(descending ? C - 1 - k : k)), d = make_uint4(0, 0, 0, 0);
    if (warp < (int)cr.y) d = lds4(a_sl + 16u * cr.x);
    bool landed = true;  // the warp has missed no block of entries
#pragma unroll 1
    for (int q = q0;;) {
      if (streamed) {
        a_ent = sm0 + (uint32_t)(D.o_buf + jst * D.stage_bytes) + 16u * (uint32_t)lane;
        mbar_wait(mst + 8u * (uint32_t)jst, jpar, D.err, polls);
        landed = __all_sync(0xffffffffu, polls > 0);
      }
      uint4 ncr = cr, nd = d;
      bool waited = false;
#pragma unroll 1
      for (int si = warp;;) {
        const bool any = si < (int)cr.y && landed;
        const int row0 = (int)(d.x & 0xFFFFu), row = row0 + ri, np = (int)(d.w & 1023u);
        const uint32_t ea = a_ent + 16u * d.z, a_row = a_bd + 2u * (uint32_t)sizeof(T) * (uint32_t)row;
        uint4 u[4];
        T bv, dv;
        uint32_t pa = 0, pm = 0;  // this lane's first halo store: where to, which barrier, which lane has the value
        int src = 0;
        if (any) {
          load_units(u, ea);
          lds_pair(a_row, bv, dv);
          int e;  // lanes past the list: not sent
          lds1(a_xd + 4u * ((d.w >> 10) + (uint32_t)lane), e);
          const uint32_t a = a_x + store_there(e) * (uint32_t)sizeof(T);
          pa = cl_map(a, lane < np ? store_cta(e) : 0u);
          pm = pa + (mcur() - a);  // the same CTA's window
          src = (((int)store_row(e) - row0) << lg) & 31;
        }
        if (!waited) {
          waited = true;
          if (++k == C) k = 0;
          if (q + 1 < nq) {
            ncr = lds4(a_cr + 16u * (uint32_t)(descending ? C - 1 - k : k));
            if (warp < (int)ncr.y) nd = lds4(a_sl + 16u * ncr.x);
          }
          begin();
          if (streamed) {
            issue();  // every warp has finished the step before
            stage_used();
          }
          if (!b_ready && any) lds_pair(a_row, bv, dv);
          b_ready = true;
        }
        if (any) {
          const T xn = (bv - row_sum<T>(u, ea, (int)d.y, sm0, tpr)) * dv;
          sts_if(first_part && ri < (int)(d.x >> 16), a_x + (uint32_t)sizeof(T) * (uint32_t)row, xn);
          if (np) {  // the slice's halo stores, one per lane
            cl_send_if(lane < np, pa, pm, __shfl_sync(0xffffffffu, xn, src));
            if (np > 32) {
              __syncwarp();
              push_list<T>(a_xd, (int)(d.w >> 10) + 32 + lane, (int)(d.w >> 10) + np, 32, a_x, mcur());
            }
          }
        }
        si += kClWarps;
        if (si >= (int)cr.y) break;
        d = lds4(a_sl + 16u * (cr.x + (uint32_t)(si - warp)));
      }
      end((int)cr.z);
      cr = ncr;
      d = nd;
      if (++q >= nq) break;
    }
  };

  const uint32_t a_bc = sm0 + (uint32_t)D.o_bc;
  // down the levels, and up again: one loop, so that the code of the sweeps
  // is there once
#pragma unroll 1
  for (int h = 0; h < 2 * NL; ++h) {
    const bool down = h < NL;
    const int t = down ? h : 2 * NL - 1 - h;
    if (h == NL) {
      // coarsest: x_c = A^-1 b_c, a warp per kC own rows at a time, the first
      // rows' coefficients loaded before the wait (they come from L2, so many have
      // to be in flight); sums in the coefficients' type
      {
        const ClusterLevel<T>& L = D.lv[NL];
        char* img = sm + L.o_img;
        const int nown = reinterpret_cast<const int*>(img)[0], nxd = reinterpret_cast<const int*>(img)[9];
        const int* gid = reinterpret_cast<const int*>(img + L.i_cr);
        const int bytes = *reinterpret_cast<const int*>(img + L.i_ex);
        const uint32_t a_xd = sm0 + (uint32_t)(L.o_img + L.i_xd), a_x = sm0 + (uint32_t)L.o_x;
        constexpr bool kWiden = sizeof(A) > sizeof(T);
        // rows at a time and coefficients of each that a lane holds (and loads
        // before the wait): as many as the registers take without spills.
        // Columns past 32 kA are loaded as they are added, which a wait for L2
        // each 128 columns makes dear: with kA = 12 the solve on the 250x122
        // torus (761 columns) took 892 us for 822, the bi-Laplacian 2407 for
        // 2267; two rows at a time measure as four
        constexpr int kC = sizeof(A) == 4 ? 4 : 1, kA = 24;
        const uint32_t a_rhs = kWiden ? sm0 + (uint32_t)D.o_bd : a_bc;
        const int n = D.nc;
        A a[kC][kA];
        auto coefs = [&](int i) {
#pragma unroll
          for (int c = 0; c < kC; ++c) {
            const A* ar = ainv + (int64_t)gid[i + c < nown ? i + c : i] * n;
#pragma unroll
            for (int q = 0; q < kA; ++q) a[c][q] = lane + 32 * q < n ? ar[lane + 32 * q] : A(0);
          }
        };
        int i = warp * kC;
        if (i < nown) coefs(i);
        begin();
        mbar_wait(mbc, 0u, D.err, polls);
        if constexpr (kWiden) {  // the right-hand side in FP64, once for all rows
          for (int j = tid; j < n; j += kClThreads) {
            T bv;
            lds1(a_bc + (uint32_t)sizeof(T) * (uint32_t)j, bv);
            sts(a_rhs + 8u * (uint32_t)j, to_f64(bv));
          }
          __syncthreads();
        }
#pragma unroll 1
        while (i < nown) {
          A acc[kC];
#pragma unroll
          for (int c = 0; c < kC; ++c) acc[c] = 0;
#pragma unroll
          for (int q = 0; q < kA; ++q) {
            A bv = 0;
            if (lane + 32 * q < n) lds1(a_rhs + (uint32_t)sizeof(A) * (uint32_t)(lane + 32 * q), bv);
#pragma unroll
            for (int c = 0; c < kC; ++c) acc[c] += a[c][q] * bv;
          }
          if (n > 32 * kA)
#pragma unroll 1
            for (int c = 0; c < kC; ++c) {
              const A* ar = ainv + (int64_t)gid[i + c < nown ? i + c : i] * n;
              A t = 0;
#pragma unroll 4
              for (int q = lane + 32 * kA; q < n; q += 32) {
                A bv;
                lds1(a_rhs + (uint32_t)sizeof(A) * (uint32_t)q, bv);
                t += ar[q] * bv;
              }
              acc[c] += t;
            }
          const int cur = i;
          i += kClWarps * kC;
          if (i < nown) coefs(i);
#pragma unroll
          for (int c = 0; c < kC; ++c) {
#pragma unroll 1
            for (int o = 16; o > 0; o >>= 1) acc[c] += __shfl_xor_sync(0xffffffffu, acc[c], o);
            if (lane == c && cur + c < nown) {
              const uint32_t xc = a_x + (uint32_t)sizeof(T) * (uint32_t)(cur + c);
              if constexpr (kWiden) sts(xc, f32_rn(acc[c]));
              else sts(xc, acc[c]);
            }
          }
        }
        __syncthreads();
        push_list<T>(a_xd, tid, nxd, kClThreads, a_x, mcur());
        end(bytes);
      }
    }
    if (!down) {  // prolongation
      const ClusterLevel<T>& L = D.lv[t];
      char* img = sm + L.o_img;
      const int* hd = reinterpret_cast<const int*>(img);
      // halo stores [lo, hi) are of rows that the post-smoothing updates first
      const int nown = hd[0], lo = hd[5], hi = hd[6], nxd = hd[9];
      const int bytes = reinterpret_cast<const int*>(img + L.i_ex)[2];
      const uint32_t a_xd = sm0 + (uint32_t)(L.o_img + L.i_xd), a_x = sm0 + (uint32_t)L.o_x;
      const uint32_t a_u = sm0 + (uint32_t)D.lv[t + 1].o_x;
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
      begin();
#pragma unroll 1
      for (int i0 = tid; i0 < nown; i0 += kP * kClThreads) {
        if (i0 != tid) weights(i0);
#pragma unroll
        for (int k = 0; k < kP; ++k) {
          const int i = i0 + k * kClThreads;
          if (i < nown) {
            T v, u[3];
            lds1(a_x + (uint32_t)sizeof(T) * (uint32_t)i, v);
#pragma unroll
            for (int m = 0; m < 3; ++m) lds1(a_u + (uint32_t)sizeof(T) * (uint32_t)id[k][m], u[m]);
            v += w[k][0] * u[0] + w[k][1] * u[1] + w[k][2] * u[2];
            sts(a_x + (uint32_t)sizeof(T) * (uint32_t)i, v);
          }
        }
      }
      __syncthreads();
      push_list<T>(a_xd, tid, lo, kClThreads, a_x, mcur());
      push_list<T>(a_xd, hi + tid, nxd, kClThreads, a_x, mcur());
      end(bytes);
    }
    const bool first_done = down && (t == 0 ? c0_first != 0 : D.nu_pre > 0);
    sweeps(t, first_done ? 1 : 0, (down ? D.nu_pre : D.nu_post) * D.lv[t].ncolor, !down && !D.post_forward,
           t == 0 || !down);
    if (!down) continue;
    const ClusterLevel<T>& L = D.lv[t];
    const ClusterLevel<T>& N = D.lv[t + 1];
    char* img = sm + L.o_img;
    const int* hd = reinterpret_cast<const int*>(img);
    const int* ex = reinterpret_cast<const int*>(img + L.i_ex);  // residual, restriction, prolongation
    const int C = L.ncolor;
    // the residual's buffer alternates between the levels: without
    // pre-smoothing a level's residual follows the finer one's restriction
    const uint32_t a_r = sm0 + (uint32_t)D.o_r[t & 1];
    // residual of the own rows, sent to the CTAs that restrict it
    {
      const uint32_t a_sl = sm0 + (uint32_t)(L.o_img + L.i_sl);
      const int4* cr = reinterpret_cast<const int4*>(img + L.i_cr);
      const uint32_t a_x = sm0 + (uint32_t)L.o_x, a_bd = sm0 + (uint32_t)L.o_val, a_dg = a_bd + (uint32_t)L.v_diag;
      const int tpr = L.tpr, ri = lane >> L.lg_tpr;
      uint32_t a_ent = sm0 + (uint32_t)(L.o_val + L.v_ent) + 16u * (uint32_t)lane;
      uint4 d = make_uint4(0, 0, 0, 0), u[4];
      auto load = [&](uint4& dd, uint4 (&uu)[4], int s) {
        dd = lds4(a_sl + 16u * (uint32_t)s);
        load_units(uu, a_ent + 16u * dd.z);
      };
      auto row = [&]() {
        const T acc = row_sum<T>(u, a_ent + 16u * d.z, (int)d.y, sm0, tpr);
        const uint32_t o = (uint32_t)sizeof(T) * (uint32_t)((int)(d.x & 0xFFFFu) + ri);
        T bv, dg, xv;
        lds1(a_bd + 2u * o, bv);
        lds1(a_dg + o, dg);
        lds1(a_x + o, xv);
        sts_if((lane & (tpr - 1)) == 0 && ri < (int)(d.x >> 16), a_r + o, bv - (acc + dg * xv));
      };
      if (!L.streamed) {
        int s = warp;
        const int se = hd[2];
        if (s < se) load(d, u, s);
        begin();
#pragma unroll 1
        while (s < se) {
          uint4 dn = d, un[4] = {u[0], u[1], u[2], u[3]};
          s += kClWarps;
          if (s < se) load(dn, un, s);
          row();
          d = dn;
#pragma unroll
          for (int q = 0; q < 4; ++q) u[q] = un[q];
        }
        __syncthreads();
      } else {
        // as many colours at a time as stages hold (the colours' slices follow one another)
        begin();
        issue();
#pragma unroll 1
        for (int k = 0; k < C;) {
          const int nk = C - k < NS ? C - k : NS;
#pragma unroll 1
          for (int q = 0, st = jst, par = (int)jpar; q < nk; ++q) {
            mbar_wait(mst + 8u * (uint32_t)st, (unsigned)par, D.err, polls);
            if (++st == NS) {
              st = 0;
              par ^= 1;
            }
          }
          const int se = __all_sync(0xffffffffu, polls > 0) ? cr[k + nk - 1].x + cr[k + nk - 1].y : 0;
#pragma unroll 1
          for (int s = cr[k].x + warp, q = 0; s < se; s += kClWarps) {
#pragma unroll 1
            while (s >= cr[k + q].x + cr[k + q].y) ++q;
            const int st = jst + q < NS ? jst + q : jst + q - NS;
            a_ent = sm0 + (uint32_t)(D.o_buf + st * D.stage_bytes) + 16u * (uint32_t)lane;
            load(d, u, s);
            row();
          }
          __syncthreads();
          // the stages of this group may be filled again; one issue stays for
          // the next user of the stream, which makes one when it begins
#pragma unroll 1
          for (int q = 0; q < nk; ++q) {
            stage_used();
            if (k + nk < C || q + 1 < nk) issue();
          }
          k += nk;
        }
      }
      push_list<T>(sm0 + (uint32_t)(L.o_img + L.i_rd), tid, hd[11], kClThreads, a_r, mcur());
      end(ex[0]);
    }
    // restriction b_{l+1} = P^T r over the own coarse rows; x_{l+1} is zero,
    // but the rows of colour 0 of a smoothed level take their first update
    // (b - 0) / a_ii right away.  The first weights are loaded before the wait.
    {
      const int4* rs = L.r_sl + (int64_t)cta * L.rsl_max;
      const int nrs = hd[3], tpr = L.r_tpr, lg = L.lg_r_tpr;
      const uint16_t* rcol = L.r_col + (int64_t)cta * L.r_max;
      const T* rw = L.r_w + (int64_t)cta * L.r_max;
      constexpr int kR = 16;
      T wv[kR];
      int ci[kR];
      int w = 0, row = 0, e = 0;
      bool lead = false;
      auto terms = [&](int q0) {
#pragma unroll
        for (int q = 0; q < kR; ++q) {
          wv[q] = q0 + q < w ? rw[e + (q0 + q) * 32] : T(0);
          ci[q] = q0 + q < w ? rcol[e + (q0 + q) * 32] : 0;
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
      char* nimg = sm + N.o_img;
      const bool first_upd = D.nu_pre > 0 && t + 1 < NL;
      const int nc0 = first_upd ? reinterpret_cast<const int*>(nimg)[4] : 0;
      const uint32_t a_gid = sm0 + (uint32_t)(N.o_img + N.i_cr);  // coarsest level: global rows of the own rows
      const uint32_t a_xn = sm0 + (uint32_t)N.o_x, a_bdn = sm0 + (uint32_t)N.o_val;
      begin();
#pragma unroll 1
      for (; s < nrs;) {
        T acc = 0;
#pragma unroll 1
        for (int q0 = 0; q0 < w; q0 += kR) {
          T rv[kR];
#pragma unroll
          for (int q = 0; q < kR; ++q) lds1(a_r + (uint32_t)sizeof(T) * (uint32_t)ci[q], rv[q]);
#pragma unroll
          for (int q = 0; q < kR; ++q)
            if (q0 + q < w) acc += wv[q] * rv[q];
          if (q0 + kR < w) terms(q0 + kR);
        }
#pragma unroll 1
        for (int o = 1; o < tpr; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        if (t + 1 < NL) {
          if (lead) {
            const uint32_t o = (uint32_t)sizeof(T) * (uint32_t)row;
            sts(a_bdn + 2u * o, acc);
            if (row < nc0) {
              T dv;
              lds1(a_bdn + 2u * o + (uint32_t)sizeof(T), dv);
              sts(a_xn + o, (acc - T(0)) * dv);
            }
          }
        } else if (lead) {  // the coarsest right-hand side goes to every CTA
          int gr;
          lds1(a_gid + 4u * (uint32_t)row, gr);
          const uint32_t a = a_bc + (uint32_t)sizeof(T) * (uint32_t)gr;
          sts(a, acc);
#pragma unroll 1
          for (int c = 1; c < D.ncta; ++c) {
            const uint32_t to = cl_map(a, (unsigned)(cta + c >= D.ncta ? cta + c - D.ncta : cta + c));
            cl_send(to, to + (mbc - a), acc);
          }
        }
        s += kClWarps;
        if (s < nrs) start(s);
      }
      if (first_upd) {
        __syncthreads();
        push_list<T>(sm0 + (uint32_t)(N.o_img + N.i_xd), tid, reinterpret_cast<const int*>(nimg)[10], kClThreads, a_xn, mcur());
      }
      end(ex[1]);
    }
  }
  __syncthreads();
  if (ph > 0) mbar_wait(mph + 8u * (uint32_t)((ph - 1) & 1), (unsigned)((ph - 1) >> 1) & 1u, D.err, polls);
  {
    const T* x = reinterpret_cast<const T*>(sm + D.lv[0].o_x);
#pragma unroll 1
    for (int i = tid; i < n0own; i += kClThreads) xg[l2g[i]] = x[i];
  }
  // the copies in flight land first: tables, the last block issued into every stage
  if ((tid == 0 || tid == kClThreads - 32) && polls == 0) {
    int again = kWaitPolls;
#pragma unroll 1
    for (int q = 0; q <= NL; ++q) mbar_wait(mimg + 8u * q, 0u, D.err, again);
#pragma unroll 1
    for (int q = issued > NS ? issued - NS : 0; q < issued; ++q)
      mbar_wait(mst + 8u * (uint32_t)(q % NS), (unsigned)(q / NS) & 1u, D.err, again);
  }
  cl_arrive();  // no CTA's shared memory goes before every message has landed
  cl_wait();
  if (polls == 0) linger();
}

// Element e of a job is the level's value in slot src[e] >= 0, 0 for -1, or
// vector element -2 - src[e] (1/a_ii or a_ii) below; it goes to byte
// (e / per) * cta_bytes + (e % per) * step of out.
template <class T>
struct RefreshJobs {
  int njob = 0;
  struct Job {
    int64_t n, per, cta_bytes;
    int step;
    const int32_t* src;
    const T *val, *vec;
    char* out;
  } job[3 * kClMaxLevels];
};
template <class T>
__global__ void k_cluster_values(const __grid_constant__ RefreshJobs<T> J) {
  const auto& q = J.job[blockIdx.y];
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < q.n; e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s = q.src[e];
    const T v = s >= 0 ? q.val[s] : s == -1 ? T(0) : q.vec[-2 - s];
    *reinterpret_cast<T*>(q.out + (e / q.per) * q.cta_bytes + (e % q.per) * q.step) = v;
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

// The kernel that a cluster runs.
template <class T>
auto cluster_kernel(const ClusterDesc<T>& D) {
  return D.coarse64 ? k_cluster_cycle<T, double> : k_cluster_cycle<T, T>;
}

// Whether the device can run such a cluster (sets the kernel's attributes).
template <class T>
bool cluster_fits(const ClusterDesc<T>& D) {
  auto* k = cluster_kernel(D);
  if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess ||
      cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemLimit) != cudaSuccess) {  // the limit every handle's layout stays within
    cudaGetLastError();
    return false;
  }
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg = cluster_config(D, at, nullptr);
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, k, &cfg) != cudaSuccess) {
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
  std::vector<uint16_t> ecol, rcol;  // per entry slot: unit u, lane q, slot v of the unit at (32 u + q) per + v
  std::vector<int32_t> esrc;
  std::vector<double> rw;
  std::vector<uint32_t> xp, xd, rp, rd;  // halo stores of x and of the residual
  std::vector<uint16_t> pidx;            // 3 x own
  std::vector<double> pw;
  std::vector<int> hcol, rows0;          // per colour: halo rows, first own row (+ end)
  int own0 = 0;                          // own rows of colour 0
};
struct Tab {
  int64_t n = 0;
  int ncolor = 0, tpr = 1, r_tpr = 1;
  bool wide = false;
  std::vector<int32_t> owner, local;
  std::vector<Part> part;
  std::vector<std::vector<int32_t>> partners;  // level l0 only: the CTAs each CTA exchanges messages with
  int n_own = 0, n_loc = 0, n_r = 0, nsl = 0, nrsl = 0, nxd = 0, nrd = 0, blk = 0, ent = 0, r_max = 0;  // largest over the CTAs (entries in units)
};

int lanes_per_row(double rows, double len) {
  int t = 1;
  while (t < 8 && rows * (2 * t) <= 32 * kClWarps && len >= 4.0 * t) t *= 2;
  return t;
}

// Slices of `rows` rows per slice from rows [0, n) of given lengths; emit(slice, first row, rows, width).
template <class Len, class Emit>
void cut_slices(int i0, int i1, int per, int tpr, int per_unit, bool pairs, Len len, Emit emit) {
  for (int a = i0; a < i1; a += per) {
    const int nr = std::min(per, i1 - a);
    int w = 0;
    for (int q = 0; q < nr; ++q) w = std::max(w, (len(a + q) + tpr - 1) / tpr);
    w = (w + per_unit - 1) / per_unit;
    emit(a, nr, pairs ? std::max(2, (w + 1) & ~1) : w);
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

// Host threads that build one precision's tables, started once for all the
// stages (starting a thread takes about 30 us: five stages that each started
// up to 15 spent 2 ms of 3.5 on it).
class Team {
 public:
  explicit Team(int workers) {
    th_.reserve(workers);
    for (int i = 0; i < workers; ++i) {
      try {
        th_.emplace_back([this] { serve(); });
      } catch (const std::system_error&) {
        break;  // no more threads: the others do the rest
      }
    }
  }
  ~Team() {
    {
      std::lock_guard<std::mutex> g(lock_);
      stop_ = true;
    }
    wake_.notify_all();
    for (auto& t : th_) t.join();
  }
  // Runs f(0) .. f(n - 1) on the team and the calling thread.  What a call
  // throws is thrown again here, after every call has ended.
  void run(int n, const std::function<void(int)>& f) {
    {
      std::lock_guard<std::mutex> g(lock_);
      f_ = &f;
      n_ = n;
      next_ = 0;
      err_ = nullptr;
      ++stage_;
    }
    wake_.notify_all();
    work(f, n);
    std::unique_lock<std::mutex> g(lock_);
    f_ = nullptr;  // a thread that wakes later finds nothing to do
    done_.wait(g, [this] { return busy_ == 0; });
    if (err_) std::rethrow_exception(err_);
  }

 private:
  void work(const std::function<void(int)>& f, int n) {
    try {
      for (int i = next_++; i < n; i = next_++) f(i);
    } catch (...) {
      std::lock_guard<std::mutex> g(lock_);
      err_ = std::current_exception();
    }
  }
  void serve() {
    std::unique_lock<std::mutex> g(lock_);
    for (unsigned seen = 0;;) {
      wake_.wait(g, [&] { return stop_ || stage_ != seen; });
      if (stop_) return;
      seen = stage_;
      if (!f_) continue;
      const std::function<void(int)>* f = f_;
      const int n = n_;
      ++busy_;
      g.unlock();
      work(*f, n);
      g.lock();
      if (--busy_ == 0) done_.notify_all();
    }
  }
  std::vector<std::thread> th_;
  std::mutex lock_;
  std::condition_variable wake_, done_;
  const std::function<void(int)>* f_ = nullptr;
  int n_ = 0, busy_ = 0;
  unsigned stage_ = 0;
  bool stop_ = false;
  std::atomic<int> next_{0};
  std::exception_ptr err_;
};

// The tables of levels l0 .. lambda over ncta CTAs (host); false when a CTA
// would hold too many rows.  The CTAs' parts are independent given the owners
// and local indices of the rows, and so are the levels' halo lists: they are
// built side by side.
bool build_tables(Team& team, const gmg_ctx* c, int l0, int ncta, int per_unit, const std::vector<std::vector<int64_t>>& hrp,
                  const std::vector<std::vector<int32_t>>& hcol, const std::vector<std::vector<int32_t>>& perm,
                  const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P, std::vector<Tab>& tab) {
  const int lam = c->nlev - 1, nl = lam - l0;
  tab.assign(nl + 1, Tab());
  int64_t nmax = 0;
  // transposed prolongation from level t + 1's rows (fine rows ascending)
  std::vector<std::vector<int64_t>> tptr(nl);
  std::vector<std::vector<int32_t>> tcol(nl);
  std::vector<std::vector<double>> tw(nl);
  for (int t = 0; t <= nl; ++t) nmax = std::max(nmax, c->L[l0 + t].n);
  team.run(2 * nl + 1, [&](int q) {
    if (q <= nl) {
      const int t = q;
      const Level& L = c->L[l0 + t];
      Tab& T = tab[t];
      T.n = L.n;
      T.ncolor = t < nl ? L.ncolor : 0;
      T.part.assign(ncta, Part());
      for (Part& p : T.part) p.own.reserve(L.n / ncta + 1);
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
      return;
    }
    const int t = q - nl - 1, l = l0 + t;
    const gmg_prolong& p = P[l];
    const int64_t nf = c->L[l].n, nn = c->L[l + 1].n;
    auto& cnt = tptr[t];
    cnt.assign(nn + 1, 0);
    for (int64_t r = 0; r < nf; ++r)
      for (int s = 0; s < 3; ++s)
        if (p.w[3 * r + s] != 0.0) cnt[iperm[l + 1][p.idx[3 * r + s]] + 1]++;
    for (int64_t J = 0; J < nn; ++J) cnt[J + 1] += cnt[J];
    tcol[t].resize(cnt[nn]);
    tw[t].resize(cnt[nn]);
    std::vector<int64_t> fill(cnt.begin(), cnt.end() - 1);
    for (int64_t r = 0; r < nf; ++r) {
      const int64_t old = perm[l][r];
      for (int s = 0; s < 3; ++s)
        if (p.w[3 * old + s] != 0.0) {
          const int64_t at = fill[iperm[l + 1][p.idx[3 * old + s]]]++;
          tcol[t][at] = (int32_t)r;
          tw[t][at] = p.w[3 * old + s];
        }
    }
  });
  for (int t = 0; t < nl; ++t)
    tab[t].r_tpr = tab[t].wide ? 1
                               : lanes_per_row((double)tab[t + 1].n / ncta,
                                               (double)tptr[t].back() / (double)tab[t + 1].n);
  std::atomic<bool> fits{true};
  team.run(ncta, [&](int a) {
    std::vector<int32_t> loc, stamp;
    loc.reserve(nmax);
    stamp.reserve(nmax);
    for (int t = 0; t <= nl; ++t) {
      Tab& T = tab[t];
      const int l = l0 + t;
      const int64_t *rp = hrp[l].data();
      const int32_t *ci = hcol[l].data(), *pm = perm[l].data(), *ip = iperm[l].data();
      loc.resize(T.n);  // read only where written below
      stamp.assign(T.n, 0);
      Part& p = T.part[a];
      auto see = [&](int32_t r) {
        if (T.owner[r] != a && !stamp[r]) {
          stamp[r] = 1;
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
      if ((int)(p.own.size() + p.halo.size()) >= kClMaxLocal) {
        fits = false;
        return;
      }
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
      if (t == nl) continue;
      // entries in the order of the level's sliced ELL, tpr lanes per row
      const Level& L = c->L[l];
      const int per = 32 / T.tpr;
      auto len = [&](int i) { return (int)(rp[pm[p.own[i]] + 1] - rp[pm[p.own[i]]] - 1); };
      const size_t guess = (size_t)(1.25 * (double)(L.nnz - L.n) / ncta);
      p.ecol.reserve(guess);
      p.esrc.reserve(guess);
      int i0 = 0;
      for (int k = 0; k < T.ncolor; ++k) {
        p.csl.push_back((int32_t)p.sl.size());
        p.blk.push_back((int32_t)(p.ecol.size() / per_unit));
        p.rows0.push_back(i0);
        int i1 = i0;
        while (i1 < (int)p.own.size() && p.own[i1] < L.color_off[k + 1]) ++i1;
        cut_slices(i0, i1, per, T.tpr, per_unit, true, len, [&](int r0, int nr, int w) {
          const size_t base = p.ecol.size();  // entry slots before this slice
          p.sl.push_back({r0 | (nr << 16), w, (int32_t)(base / per_unit), 0});
          p.ecol.resize(base + 32 * (size_t)w * per_unit, 0);
          p.esrc.resize(base + 32 * (size_t)w * per_unit, -1);
          for (int q = 0; q < nr; ++q) {
            const int32_t r = p.own[r0 + q];
            const int64_t old = pm[r];
            const int64_t slice = L.color_slice_off[k] + (r - L.color_off[k]) / kSlice;
            int64_t slot = L.h_ptr[slice] + (r - L.color_off[k]) % kSlice;
            // entry m of the row: lane part m mod tpr, unit (m / tpr) / per_unit, slot (m / tpr) % per_unit
            auto at_slot = [&](int m) {
              const int u = m / T.tpr;
              return base + (32 * (size_t)(u / per_unit) + q * T.tpr + m % T.tpr) * per_unit + u % per_unit;
            };
            int m = 0;
            for (int64_t e = rp[old]; e < rp[old + 1]; ++e) {
              if (ci[e] == old) continue;
              const size_t g = at_slot(m);
              p.ecol[g] = (uint16_t)at(ip[ci[e]]);
              p.esrc[g] = (int32_t)slot;
              slot += kSlice;
              ++m;
            }
            for (; m < T.tpr * w * per_unit; ++m) p.ecol[at_slot(m)] = (uint16_t)(r0 + q);  // padding: itself, value 0
          }
        });
        i0 = i1;
      }
      p.csl.push_back((int32_t)p.sl.size());
      p.blk.push_back((int32_t)(p.ecol.size() / per_unit));
      p.rows0.push_back(i0);
      p.hcol.assign(T.ncolor, 0);
      int k = 0;
      for (int32_t r : p.halo) {  // ascending: colour by colour
        while (r >= L.color_off[k + 1]) ++k;
        p.hcol[k]++;
      }
      // restriction: the own coarse rows gather the residual (fine rows ascending)
      const std::vector<int64_t>& cnt = tptr[t];
      const std::vector<int32_t>& tc = tcol[t];
      const std::vector<int32_t>& coarse = tab[t + 1].part[a].own;
      stamp.assign(T.n, 0);
      for (int32_t J : coarse)
        for (int64_t q = cnt[J]; q < cnt[J + 1]; ++q)
          if (T.owner[tc[q]] != a && !stamp[tc[q]]) {
            stamp[tc[q]] = 1;
            p.rhalo.push_back(tc[q]);
          }
      std::sort(p.rhalo.begin(), p.rhalo.end());
      if ((int)(p.own.size() + p.rhalo.size()) >= kClMaxLocal) {
        fits = false;
        return;
      }
      for (size_t q = 0; q < p.rhalo.size(); ++q) loc[p.rhalo[q]] = (int32_t)(p.own.size() + q);
      auto rlen = [&](int i) { return (int)(cnt[coarse[i] + 1] - cnt[coarse[i]]); };
      cut_slices(0, (int)coarse.size(), 32 / T.r_tpr, T.r_tpr, 1, false, rlen, [&](int r0, int nr, int w) {
        const size_t base = p.rcol.size();
        p.rsl.push_back({r0 | (nr << 16), w, (int32_t)base, 0});
        p.rcol.resize(base + 32 * (size_t)w, 0);
        p.rw.resize(base + 32 * (size_t)w, 0.0);
        for (int q = 0; q < nr; ++q) {
          int m = 0;
          for (int64_t e = cnt[coarse[r0 + q]]; e < cnt[coarse[r0 + q] + 1]; ++e, ++m) {
            const size_t g = base + 32 * (size_t)(m / T.r_tpr) + q * T.r_tpr + m % T.r_tpr;
            p.rcol[g] = (uint16_t)(T.owner[tc[e]] == a ? T.local[tc[e]] : loc[tc[e]]);
            p.rw[g] = tw[t][e];
          }
        }
      });
    }
  });
  if (!fits) return false;
  team.run(2 * nl + 1, [&](int q) {
    Tab& T = tab[q / 2];
    push_lists(T.owner, T.local, T.part, q % 2 != 0);
  });
  // partners: the CTAs that send a CTA values on some level, or that it sends to
  std::vector<char> ex((size_t)ncta * ncta, 0);
  for (int t = 0; t <= nl; ++t)
    for (int a = 0; a < ncta; ++a)
      for (const auto* h : {&tab[t].part[a].halo, &tab[t].part[a].rhalo})
        for (int32_t r : *h) ex[a * ncta + tab[t].owner[r]] = ex[tab[t].owner[r] * ncta + a] = 1;
  tab[0].partners.assign(ncta, {});
  for (int a = 0; a < ncta; ++a)
    for (int b = 0; b < ncta; ++b)
      if (a != b && ex[a * ncta + b]) tab[0].partners[a].push_back(b);
  for (Tab& T : tab)
    for (Part& p : T.part) {
      T.n_own = std::max(T.n_own, (int)p.own.size());
      T.n_loc = std::max(T.n_loc, (int)(p.own.size() + p.halo.size()));
      T.n_r = std::max(T.n_r, (int)(p.own.size() + p.rhalo.size()));
      T.nsl = std::max(T.nsl, (int)p.sl.size());
      T.nrsl = std::max(T.nrsl, (int)p.rsl.size());
      T.nxd = std::max(T.nxd, (int)p.xd.size());
      T.nrd = std::max(T.nrd, (int)p.rd.size());
      T.ent = std::max(T.ent, (int)(p.ecol.size() / per_unit));
      T.r_max = std::max(T.r_max, (int)p.rcol.size());
      for (size_t k = 0; k + 1 < p.blk.size(); ++k) T.blk = std::max(T.blk, p.blk[k + 1] - p.blk[k]);
    }
  return true;
}

// Every index the kernel uses: columns and halo stores in range, each halo
// copy written by its row's owner exactly once, slices covering the rows.
bool check_level(const std::vector<Tab>& tab, int per_unit, int t) {
  const int nl = (int)tab.size() - 1;
  {
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
              ((size_t)s.z + 32 * (size_t)s.y) * per_unit > p.ecol.size())
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

bool check_tables(Team& team, const std::vector<Tab>& tab, int per_unit) {
  std::atomic<bool> ok{true};
  team.run((int)tab.size(), [&](int t) {
    if (!check_level(tab, per_unit, t)) ok = false;
  });
  return ok;
}

int64_t al16(int64_t v) { return (v + 15) & ~(int64_t)15; }

// Shared-memory layout: resident levels' entries in shared memory where
// everything fits, the largest levels' entries streamed where not (three
// stages at least, two as a last resort).  False when nothing fits.
template <class T>
bool lay_out(const std::vector<Tab>& tab, int nu_pre, int nu_post, ClusterDesc<T>& D) {
  const int nl = (int)tab.size() - 1;
  std::vector<char> streamed(nl, 0);
  int npart = 0;
  for (const auto& p : tab[0].partners) npart = std::max(npart, (int)p.size());
  for (;;) {
    int64_t cur = 0, blk = 0;
    int nsteps = 0;
    for (int t = 0; t < nl; ++t)
      if (streamed[t]) {
        nsteps += (nu_pre + 1 + nu_post) * tab[t].ncolor;  // an upper bound: a skipped first phase has no step
        blk = std::max<int64_t>(blk, tab[t].blk);
      }
    D.stage_bytes = (int)(16 * blk);
    D.o_mbar = 0;
    D.o_tok = (int)al16(8 * (kClMaxLevels + 1 + kClStages + 3));
    cur = D.o_tok + 64;
    int64_t nr[2] = {1, 1};
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
      L.r_max = std::max(32, A.r_max);
      // image: header, slices, colour records (the coarsest level: global rows), halo stores, steps, partners
      int64_t o = 64;
      L.i_ex = (int)o;
      o += 16;
      L.i_sl = (int)o;
      o += 16 * (int64_t)A.nsl;
      L.i_cr = (int)o;
      o = al16(o + (t < nl ? 16 * (int64_t)A.ncolor : 4 * (int64_t)L.n_own_max));
      L.i_xd = (int)o;
      o = al16(o + 4 * (int64_t)A.nxd);
      L.i_rd = (int)o;
      if (t < nl) o = al16(o + 4 * (int64_t)A.nrd);
      if (t == 0) {
        D.i_partners = (int)o;
        o = al16(o + 4 * (int64_t)npart);
        D.i_steps = (int)o;
        o = al16(o + 8 * (int64_t)nsteps);
      }
      L.img_bytes = (int)o;
      // values: pairs (b, 1/a_ii), a_ii, resident entries
      L.v_diag = (int)al16(2 * (int64_t)sizeof(T) * L.n_own_max);
      L.v_ent = (int)(L.v_diag + al16((int64_t)sizeof(T) * L.n_own_max));
      const int64_t vb = t < nl ? L.v_ent + (res ? 16 * (int64_t)A.ent : 0) : 0;
      if (vb > kSmemLimit || o > kSmemLimit) {
        cur = kSmemLimit + 1;
        break;
      }
      L.val_bytes = (int)vb;
      L.o_img = (int)cur;
      cur += L.img_bytes;
      L.o_val = (int)cur;
      cur += L.val_bytes;
      L.o_x = (int)cur;
      cur = al16(cur + (int64_t)sizeof(T) * L.n_loc_max);
      if (t < nl) nr[t & 1] = std::max<int64_t>(nr[t & 1], A.n_r);
    }
    for (int q = 0; q < 2; ++q) {
      D.o_r[q] = (int)std::min<int64_t>(cur, INT32_MAX);
      cur = al16(cur + (int64_t)sizeof(T) * nr[q]);
    }
    D.o_bc = (int)std::min<int64_t>(cur, INT32_MAX);
    cur = al16(cur + (int64_t)sizeof(T) * tab[nl].n);
    D.o_bd = (int)std::min<int64_t>(cur, INT32_MAX);
    if (D.coarse64 && sizeof(T) == 4) cur = al16(cur + 8 * tab[nl].n);
    D.o_buf = (int)std::min<int64_t>(cur, INT32_MAX);
    D.nsteps = nsteps;
    const bool all = std::all_of(streamed.begin(), streamed.end(), [](char v) { return v != 0; });
    // a lane loads up to two units (1 KB of a warp) past its row's
    const int64_t need = (blk == 0 ? 0 : (all ? 2 : 3) * 16 * blk) + kClSlack;
    if (cur + need <= kSmemLimit) {
      D.nstage = blk == 0 ? 0 : (int)std::min<int64_t>(kClStages, (kSmemLimit - kClSlack - cur) / D.stage_bytes);
      D.smem = (int)(cur + (int64_t)D.nstage * D.stage_bytes + kClSlack);
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

// Device arrays of one handle's tables, gathered in one host buffer so that
// they take one allocation and one copy: the arrays are declared with add(),
// then at() gives their places in the buffer.
struct Blob {
  std::vector<char> h;
  size_t size = 0;
  std::vector<std::pair<const void**, size_t>> ptrs;
  template <class U>
  size_t add(const U** d, size_t n) {  // n elements, zeroed
    const size_t o = (size + 255) & ~(size_t)255;
    size = o + std::max<size_t>(n, 1) * sizeof(U);
    ptrs.push_back({reinterpret_cast<const void**>(d), o});
    return o;
  }
  template <class U>
  U* at(size_t o) {
    return reinterpret_cast<U*>(h.data() + o);
  }
  gmg_status upload(Arena& a) {
    char* p;
    GMG_TRY(a.alloc(&p, h.size()));
    GMG_CK(cudaMemcpy(p, h.data(), h.size(), cudaMemcpyHostToDevice));
    for (auto& q : ptrs) *q.first = p + q.second;
    return GMG_OK;
  }
};

// Entry units of one part: the x addresses (byte offsets into shared memory); the values come with every refresh.
template <class T>
void fill_units(const Part& p, int o_x, char* out) {
  for (size_t e = 0; e < p.ecol.size(); ++e) {
    const uint32_t off = (uint32_t)o_x + (uint32_t)sizeof(T) * p.ecol[e];
    std::memcpy(out + (sizeof(T) == 4 ? 8 * e + 4 : 16 * e + 8), &off, 4);
  }
}

// The first halo store of the rows from local row i on.
int32_t first_store(const Part& p, int i) {
  return i < (int)p.xp.size() ? (int32_t)(p.xp[i] >> 4) : (int32_t)p.xd.size();
}

// Lays the tables of `tab` out as D says and uploads them.
template <class T>
gmg_status upload_tables(Team& team, gmg_ctx* c, const std::vector<Tab>& tab, ClusterDesc<T>& D) {
  constexpr size_t pu = sizeof(T) == 4 ? 2 : 1;  // entries per unit
  const int nl = (int)tab.size() - 1, ncta = D.ncta;
  Blob B;
  // streamed entries of all levels, CTA after CTA
  std::vector<std::vector<uint32_t>> s_off(nl);  // per level and CTA: first unit
  size_t units = 0;
  for (int t = 0; t < nl; ++t)
    if (D.lv[t].streamed)
      for (const Part& p : tab[t].part) {
        s_off[t].push_back((uint32_t)units);
        units += p.ecol.size() / pu;
      }
  for (int t = 0; t < nl; ++t)
    if (D.lv[t].streamed)
      for (const Part& p : tab[t].part) D.lv[t].n_stream += (int64_t)p.esrc.size();
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
  D.nsteps = (int)(steps[0].size() / 2);
  const size_t o_ent = B.add(&D.s_ent, units), o_src = B.add(&D.s_src, units * pu);
  struct Off {
    size_t img, vi, ds, vs, rsl, rc, rw, pi, pw;
  };
  std::vector<Off> off(nl + 1);
  size_t o_l2g = 0;
  for (int t = 0; t <= nl; ++t) {
    ClusterLevel<T>& L = D.lv[t];
    const size_t no = (size_t)ncta * L.n_own_max;
    off[t].img = B.add(&L.img, (size_t)ncta * L.img_bytes);
    if (t == 0) o_l2g = B.add(&D.l2g, (size_t)ncta * L.n_loc_max);
    if (t == nl) break;
    const int64_t ent = L.streamed ? 0 : (int64_t)tab[t].ent * pu;
    L.n_ent = ent;
    L.nvsrc = ncta * ent;
    off[t].vi = B.add(&L.vimg, (size_t)ncta * L.val_bytes);
    off[t].ds = B.add(&L.dsrc, no);
    off[t].vs = B.add(&L.vsrc, (size_t)L.nvsrc);
    off[t].rsl = B.add(&L.r_sl, (size_t)ncta * L.rsl_max);
    off[t].rc = B.add(&L.r_col, (size_t)ncta * L.r_max);
    off[t].rw = B.add(&L.r_w, (size_t)ncta * L.r_max);
    off[t].pi = B.add(&L.p_idx, 3 * no);
    off[t].pw = B.add(&L.p_w, 3 * no);
  }
  B.h.resize(B.size);
  // each CTA's part of every array
  team.run(ncta, [&](int q) {
    for (int t = 0; t <= nl; ++t) {
      const Tab& A = tab[t];
      const ClusterLevel<T>& L = D.lv[t];
      const Part& p = A.part[q];
      const size_t S = sizeof(T), no = (size_t)L.n_own_max, m = p.own.size();
      char* base = B.at<char>(off[t].img) + (size_t)q * L.img_bytes;
      auto put = [&](int at, const void* v, size_t bytes) {
        if (bytes) std::memcpy(base + at, v, bytes);
      };
      int32_t hd[16] = {(int32_t)m, (int32_t)(m + p.halo.size()), (int32_t)p.sl.size(), (int32_t)p.rsl.size(), p.own0};
      hd[9] = (int32_t)p.xd.size();
      int32_t ex[4] = {0, 0, 0, 0};  // halo bytes that the residual, restriction, prolongation brings (coarsest: the solve)
      if (t < nl) {
        const int kf = D.post_forward ? 0 : A.ncolor - 1;  // the colour that the post-smoothing updates first
        hd[5] = first_store(p, D.nu_post > 0 ? p.rows0[kf] : 0);
        hd[6] = first_store(p, D.nu_post > 0 ? p.rows0[kf + 1] : 0);
        hd[10] = first_store(p, p.own0);
        hd[11] = (int32_t)p.rd.size();
        for (int k = 0; k < A.ncolor; ++k) {  // first slice, slices, halo bytes of the colour's phase
          const int32_t rec[4] = {p.csl[k], p.csl[k + 1] - p.csl[k], (int32_t)(S * p.hcol[k]), 0};
          put(L.i_cr + 16 * k, rec, 16);
        }
        ex[0] = (int32_t)(S * p.rhalo.size());
        if (D.nu_pre > 0 && t + 1 < nl) ex[1] = (int32_t)(S * tab[t + 1].part[q].hcol[0]);
        ex[2] = (int32_t)(S * (p.halo.size() - (D.nu_post > 0 ? p.hcol[kf] : 0)));
      } else {
        ex[0] = (int32_t)(S * p.halo.size());
      }
      if (t == 0) {
        hd[7] = (int32_t)A.partners[q].size();
        hd[8] = (int32_t)tab[nl].part[q].own.size();
        put(D.i_partners, A.partners[q].data(), 4 * A.partners[q].size());
        put(D.i_steps, steps[q].data(), 4 * steps[q].size());
        int32_t* l2g = B.at<int32_t>(o_l2g) + (size_t)q * L.n_loc_max;
        std::copy(p.own.begin(), p.own.end(), l2g);
        std::copy(p.halo.begin(), p.halo.end(), l2g + m);
      }
      put(0, hd, sizeof(hd));
      put(L.i_ex, ex, sizeof(ex));
      put(L.i_sl, p.sl.data(), p.sl.size() * sizeof(Slice));
      if (t == nl) put(L.i_cr, p.own.data(), m * 4);
      // halo stores in row order
      auto put_list = [&](int at, const std::vector<uint32_t>& lp, const std::vector<uint32_t>& ld) {
        uint32_t* o = reinterpret_cast<uint32_t*>(base + at);
        for (size_t i = 0; i < lp.size(); ++i)
          for (uint32_t e = 0; e < (lp[i] & 15u); ++e) {
            const uint32_t d = ld[(lp[i] >> 4) + e];  // CTA << 16 | local index there
            *o++ = (d >> 16) << 28 | (d & 0xFFFFu) << 14 | (uint32_t)i;
          }
      };
      put_list(L.i_xd, p.xp, p.xd);
      if (t < nl) put_list(L.i_rd, p.rp, p.rd);
      Slice* sl = reinterpret_cast<Slice*>(base + L.i_sl);
      if (L.streamed)  // entry offsets within the colour's block
        for (int k = 0; k < A.ncolor; ++k)
          for (int s = p.csl[k]; s < p.csl[k + 1]; ++s) sl[s].z -= p.blk[k];
      for (size_t s = 0; s < p.sl.size(); ++s) {  // the slices' halo stores
        const int r0 = p.sl[s].x & 0xFFFF, r1 = r0 + (p.sl[s].x >> 16);
        sl[s].w = (first_store(p, r0) << 10) | (first_store(p, r1) - first_store(p, r0));
        sl[s].y /= 2;  // pairs of units
      }
      if (t == nl) continue;
      int32_t* ds = B.at<int32_t>(off[t].ds) + (size_t)q * no;
      std::fill(ds, ds + no, -1);
      for (size_t i = 0; i < m; ++i) ds[i] = -2 - p.own[i];
      if (L.streamed) {
        fill_units<T>(p, L.o_x, B.at<char>(o_ent) + 16 * (size_t)s_off[t][q]);
        std::copy(p.esrc.begin(), p.esrc.end(), B.at<int32_t>(o_src) + pu * (size_t)s_off[t][q]);
      } else {
        char* u = B.at<char>(off[t].vi) + (size_t)q * L.val_bytes + L.v_ent;
        const uint32_t pad = (uint32_t)L.o_x;  // units past a CTA's own are never read; give them a valid address
        for (size_t e = p.ecol.size(); e < (size_t)A.ent * pu; ++e)
          std::memcpy(u + (pu == 2 ? 8 * e + 4 : 16 * e + 8), &pad, 4);
        fill_units<T>(p, L.o_x, u);
        int32_t* vs = B.at<int32_t>(off[t].vs) + (size_t)q * L.n_ent;
        std::fill(std::copy(p.esrc.begin(), p.esrc.end(), vs), vs + L.n_ent, -1);
      }
      std::copy(p.rsl.begin(), p.rsl.end(), B.at<Slice>(off[t].rsl) + (size_t)q * L.rsl_max);
      std::copy(p.rcol.begin(), p.rcol.end(), B.at<uint16_t>(off[t].rc) + (size_t)q * L.r_max);
      T* rw = B.at<T>(off[t].rw) + (size_t)q * L.r_max;
      for (size_t e = 0; e < p.rw.size(); ++e) rw[e] = (T)p.rw[e];
      for (int s = 0; s < 3; ++s) {
        std::copy(p.pidx.begin() + s * m, p.pidx.begin() + (s + 1) * m,
                  B.at<uint16_t>(off[t].pi) + ((size_t)q * 3 + s) * no);
        T* pw = B.at<T>(off[t].pw) + ((size_t)q * 3 + s) * no;
        for (size_t i = 0; i < m; ++i) pw[i] = (T)p.pw[s * m + i];
      }
    }
  });
  return B.upload(c->arena);
}

// The host tables of one precision's cluster (plan.l0 stays -1: none).
template <class T>
struct Plan {
  std::unique_ptr<Team> team;
  std::vector<Tab> tab;
  ClusterDesc<T> D;
  bool checked = true;
};

// Whether the coarsest solve of FP32 cycles takes the FP32 copy of the inverse
// and FP32 sums: hierarchies of two or more smoothed levels the last of which
// is small (vectors of all its rows and a CTA's share of its entries within
// one CTA's shared memory: some 6,000 rows).  Elsewhere, on two-level
// hierarchies above all, it takes the FP64 inverse with FP64 sums, as the
// launch-per-phase form does: with one smoothed level the coarsest solve is
// the whole coarse correction, and on a nearly singular system (condition
// number of the coarsest operator above 2^24) the FP32 inverse made solves
// stall (a 642-vertex sphere, (S + 1e-7 M) x = M y to 1e-7: 12 steps for 6).
// The price is the narrow FP64 pipe: 402 rows take 4.5 us more a cycle
// (2,562-vertex sphere, FP32-PCG: 252 -> 278 us).
inline bool coarsest_in_fp32(const gmg_ctx* c) {
  const int lam = c->nlev - 1;
  if (lam < 2) return false;
  const Level& L = c->L[lam - 1];
  const int64_t bytes = 24 * L.n + L.A.entries * 8 / 16 * 11 / 10 + 8 * c->L[lam].n;
  return bytes <= kSmemLimit;
}

// Whether level l takes no part in a cluster of ncta CTAs whatever fits.
inline bool too_large(const gmg_ctx* c, int l, int ncta) {
  const Level& L = c->L[l];
  const int64_t parts = std::max(1, L.ncolor) * (int64_t)ncta;
  return (L.nnz - L.n) / parts > kClPhaseEntries || (c->cl_small && L.n / parts >= kClWide) || L.A.entries > INT32_MAX;
}
inline std::vector<int> cluster_sizes(const gmg_ctx* c) {
  return c->cl_ctas > 0 ? std::vector<int>{c->cl_ctas} : std::vector<int>{16, 8};
}

template <class T>
void plan_one(const gmg_ctx* c, const std::vector<std::vector<int64_t>>& hrp,
              const std::vector<std::vector<int32_t>>& hcol, const std::vector<std::vector<int32_t>>& perm,
              const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P, Plan<T>& plan) {
  const int lam = c->nlev - 1;
  if (lam < 1 || c->cl_off) return;
  for (int ncta : cluster_sizes(c)) {
    if (ncta > 16) continue;
    for (int l0 = std::max(0, lam - kClMaxLevels); l0 < lam; ++l0) {
      // a quick lower bound of the shared memory before the tables are built
      constexpr int pu = sizeof(T) == 4 ? 2 : 1;
      int64_t least = (int64_t)sizeof(T) * c->L[lam].n, stage = 0, ent = 0;
      bool skip = false;
      for (int l = l0; l < lam; ++l) {
        const Level& L = c->L[l];
        skip = skip || too_large(c, l, ncta);
        // x, b, 1/a_ii and a_ii of the rows; entries in shared memory, or two stages of a phase
        least += (L.n / ncta) * (int64_t)(4 * sizeof(T)) + (l == l0 ? (int64_t)sizeof(T) * (L.n / ncta) : 0);
        const int64_t e = (L.nnz - L.n) * (16 / pu) / ncta;
        ent += e;
        stage = std::max(stage, 2 * e / std::max(1, L.ncolor));
      }
      if (skip || least + std::min(ent, stage) > kSmemLimit) continue;
      std::vector<Tab>& tab = plan.tab;
      if (!plan.team) {  // a thread for some 20,000 entries, four in all where that is less
        int64_t entries = 0;
        for (int l = l0; l < lam; ++l) entries += c->L[l].nnz;
        const int hw = (int)std::max(1u, std::min(16u, std::thread::hardware_concurrency()));
        plan.team.reset(new Team((int)std::min<int64_t>(hw, std::max<int64_t>(4, entries / 20000)) - 1));
      }
      Team& team = *plan.team;
      if (!build_tables(team, c, l0, ncta, pu, hrp, hcol, perm, iperm, P, tab)) continue;
      // where the ranks are not local (random order: 11-13 halo stores per
      // row on a kNN cloud) a phase would store nearly every row into every CTA
      bool local = true;
      for (int t = 0; t < lam - l0; ++t) {
        int64_t stores = 0;
        for (const Part& p : tab[t].part) stores += (int64_t)p.xd.size();
        local = local && (!tab[t].wide || stores <= 3 * tab[t].n);
      }
      if (!local) continue;
      // a CTA that waits no more may send all of a cycle's messages before a
      // partner has taken the first: they have to stay within the 2^20 - 1
      // bytes that a barrier counts (each halo row once a sweep and once or
      // twice besides, the residual's halo once, a token of 4 bytes a phase
      // from each of 15 partners)
      double bytes = 0;
      for (const Tab& t : tab) {
        size_t halo = 0, rhalo = 0;
        for (const Part& p : t.part) halo = std::max(halo, p.halo.size()), rhalo = std::max(rhalo, p.rhalo.size());
        const double nu = (double)c->opt.nu_pre + c->opt.nu_post;
        bytes += (nu + 2) * (double)(sizeof(T) * halo) + (double)(sizeof(T) * rhalo) + 60 * (nu * t.ncolor + 4);
      }
      if (bytes >= 1048575.0) continue;
      ClusterDesc<T> E{};
      E.l0 = l0;
      E.ncta = ncta;
      E.nlev = lam - l0;
      E.nc = (int)c->L[lam].n;
      E.nu_pre = c->opt.nu_pre;
      E.nu_post = c->opt.nu_post;
      E.post_forward = c->opt.post_forward;
      E.coarse64 = sizeof(T) == 8 || !coarsest_in_fp32(c);
      if (!lay_out(tab, E.nu_pre, E.nu_post, E)) continue;
      if (!check_tables(team, tab, pu)) {
        plan.checked = false;
        return;
      }
      if (!cluster_fits(E)) break;  // this cluster size cannot be scheduled: try the next
      for (int t = 0; t < E.nlev; ++t) E.wide[t] = tab[t].wide;
      plan.D = E;
      return;
    }
  }
}

template <class T>
gmg_status finish_one(gmg_ctx* c, Plan<T>& plan) {
  if (!plan.checked) {
    set_error("internal: cluster tables failed their host check");
    return GMG_ERR_INVALID_ARG;
  }
  if (plan.D.l0 < 0) return GMG_OK;
  plan.D.ainv = Src<T>::ainv(c);
  plan.D.ainv64 = c->Ainv;
  plan.D.err = c->dstatus + 3;
  plan.D.polls = c->wait_polls < 0 ? kWaitPolls : c->wait_polls;
  GMG_TRY(upload_tables(*plan.team, c, plan.tab, plan.D));
  Src<T>::desc(c) = plan.D;
  if (const char* e = std::getenv("GMG_VERBOSE"))
    if (e[0] == '1')
      std::fprintf(stderr, "gmg: FP%d cluster: from level %d, %d CTAs, %d stages, %d bytes of shared memory\n",
                   8 * (int)sizeof(T), plan.D.l0, plan.D.ncta, plan.D.nstage, plan.D.smem);
  return GMG_OK;
}

template <class T>
gmg_status refresh_one(gmg_ctx* c, cudaStream_t s) {
  ClusterDesc<T>& D = Src<T>::desc(c);
  if (D.l0 < 0) return GMG_OK;
  RefreshJobs<T> J;
  const int step = sizeof(T) == 4 ? 8 : 16;
  int64_t most = 1, off = 0;
  for (int t = 0; t < D.nlev; ++t) {
    Level& L = c->L[D.l0 + t];
    const ClusterLevel<T>& C = D.lv[t];
    const T* v = Vec<T>::v(L.A);
    char* out = const_cast<char*>(C.vimg);
    const int64_t nd = (int64_t)D.ncta * C.n_own_max;
    J.job[J.njob++] = {nd, C.n_own_max, C.val_bytes, 2 * (int)sizeof(T), C.dsrc, v, Vec<T>::dinv(L), out + sizeof(T)};
    J.job[J.njob++] = {nd, C.n_own_max, C.val_bytes, (int)sizeof(T), C.dsrc, v, Vec<T>::diag(L), out + C.v_diag};
    if (C.streamed) {
      char* ent = reinterpret_cast<char*>(const_cast<uint4*>(D.s_ent)) + off * step;
      J.job[J.njob++] = {C.n_stream, std::max<int64_t>(1, C.n_stream), 0, step, D.s_src + off, v, nullptr, ent};
      off += C.n_stream;
      most = std::max(most, C.n_stream);
    } else if (C.nvsrc > 0) {
      J.job[J.njob++] = {C.nvsrc, C.n_ent, C.val_bytes, step, C.vsrc, v, nullptr, out + C.v_ent};
      most = std::max(most, C.nvsrc);
    }
  }
  k_cluster_values<T><<<dim3((unsigned)std::min<int64_t>((most + 255) / 256, 304), (unsigned)J.njob), 256, 0, s>>>(J);
  GMG_LAUNCHED();
  return GMG_OK;
}

}  // namespace

// Whether the handle's solves run FP64 cycles.
static bool fp64_cycles(const gmg_ctx* c) {
  return c->opt.precision == GMG_FP64 || c->opt.precision == GMG_FP64_PCG;
}

// The tables being built on host threads, of either precision.  What a
// thread throws is thrown again by finish_cluster; the destructor waits for
// the threads, so the job ends before what they read does.
struct ClusterJob {
  Plan<float> p32;
  Plan<double> p64;
  std::thread th[2];
  std::exception_ptr err[2];
  template <class F>
  void run(int k, int device, F f) {
    auto body = [this, k, device, f] {
      try {
        cudaSetDevice(device);
        f();
      } catch (...) {
        err[k] = std::current_exception();
      }
    };
    try {
      th[k] = std::thread(body);
    } catch (const std::system_error&) {
      body();  // no more threads: here and now
    }
  }
  void wait() {
    for (auto& t : th)
      if (t.joinable()) t.join();
  }
  ~ClusterJob() { wait(); }
};

std::shared_ptr<ClusterJob> start_cluster(gmg_ctx* c, const std::vector<std::vector<int64_t>>& hrp,
                                          const std::vector<std::vector<int32_t>>& hcol,
                                          const std::vector<std::vector<int32_t>>& perm,
                                          const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P) {
  auto job = std::make_shared<ClusterJob>();
  ClusterJob& j = *job;
  c->cl32 = ClusterDesc<float>{};
  c->cl64 = ClusterDesc<double>{};
  if (!c->single_rhs) return job;
  auto env = [](const char* name) {
    const char* e = std::getenv(name);
    return e && e[0] == '1';
  };
  c->cl_off = env("GMG_NO_TAIL");
  c->cl_small = env("GMG_NO_CLUSTER_LEVEL");
  if (const char* e = std::getenv("GMG_TAIL_CTAS")) {
    c->cl_ctas = std::atoi(e);
    c->cl_off = c->cl_off || c->cl_ctas < 1;
  }
  c->cl32_late = fp64_cycles(c);
  if (c->cl32_late)
    j.run(1, c->device, [&, c, P] { plan_one<double>(c, hrp, hcol, perm, iperm, P, j.p64); });
  else
    j.run(0, c->device, [&, c, P] { plan_one<float>(c, hrp, hcol, perm, iperm, P, j.p32); });
  return job;
}

gmg_status finish_cluster(gmg_ctx* c, ClusterJob& job) {
  job.wait();
  for (auto& e : job.err)
    if (e) std::rethrow_exception(e);
  GMG_TRY(finish_one<float>(c, job.p32));
  return finish_one<double>(c, job.p64);
}

gmg_status late_cluster(gmg_ctx* c, cudaStream_t s, bool values) try {
  if (!c->cl32_late && !(values && fp64_cycles(c) && c->cl32.l0 >= 0)) return GMG_OK;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  bool capturing = cudaStreamIsCapturing(s, &cs) != cudaSuccess;  // the legacy stream while another one captures
  if (capturing) cudaGetLastError();
  capturing = capturing || cs != cudaStreamCaptureStatusNone;
  if (c->cl32_late) {
    if (capturing) return GMG_OK;
    const int lam = c->nlev - 1, most = cluster_sizes(c)[0];
    int lo = lam;  // the levels that may take part
    while (lo > 0 && lo > lam - kClMaxLevels && !too_large(c, lo - 1, most)) --lo;
    std::vector<std::vector<int64_t>> hrp(c->nlev);
    std::vector<std::vector<int32_t>> hcol(c->nlev), perm(c->nlev), iperm(c->nlev), pidx(c->nlev);
    std::vector<std::vector<double>> pw(c->nlev);
    std::vector<gmg_prolong> P(c->nlev);
    auto get = [](auto& v, const auto* d, int64_t n) {
      v.resize((size_t)n);
      return cudaMemcpy(v.data(), d, sizeof(v[0]) * (size_t)n, cudaMemcpyDeviceToHost);
    };
    for (int l = lo; l <= lam && lo < lam && !c->cl_off; ++l) {
      Level& L = c->L[l];
      GMG_CK(get(hrp[l], L.csr_rowptr, L.n + 1));
      GMG_CK(get(hcol[l], L.csr_col, L.nnz));
      GMG_CK(get(perm[l], L.perm, L.n));
      GMG_CK(get(iperm[l], L.iperm, L.n));
      if (l == lam) break;
      GMG_CK(get(L.h_ptr, L.A.ptr, L.A.nslice + 1));
      GMG_CK(get(pidx[l], L.p_idx_o, 3 * L.n));
      GMG_CK(get(pw[l], L.p_w_o, 3 * L.n));
      P[l] = {L.n, L.nc, pidx[l].data(), pw[l].data()};
    }
    Plan<float> plan;
    if (lo < lam) plan_one<float>(c, hrp, hcol, perm, iperm, P.data(), plan);
    for (Level& L : c->L) std::vector<int64_t>().swap(L.h_ptr);
    GMG_TRY(finish_one<float>(c, plan));
    GMG_TRY(uploads_landed());
    c->cl32_late = false;
    c->cl32_stale = c->cl32.l0 >= 0;
  }
  if (values && c->cl32_stale) {
    GMG_TRY(refresh_one<float>(c, s));
    c->cl32_stale = capturing;  // a captured launch has filled nothing yet
  } else if (values && capturing && c->cl32.l0 >= 0) {
    c->cl32_captured = true;  // replayed after refreshes without coming by here
  }
  return GMG_OK;
} catch (const std::exception& e) {
  set_error(std::string("FP32 cluster tables: ") + e.what());
  return GMG_ERR_OOM;
}

gmg_status refresh_cluster_values(gmg_ctx* c, cudaStream_t s) {
  if (fp64_cycles(c) && !c->cl32_captured) c->cl32_stale = c->cl32.l0 >= 0;
  else GMG_TRY(refresh_one<float>(c, s));
  return refresh_one<double>(c, s);
}

template <class T>
gmg_status launch_cluster(gmg_ctx* c, T* x, const T* b, bool c0_first, cudaStream_t s) {
  const ClusterDesc<T>& D = Src<T>::desc(c);
  cudaLaunchAttribute at[2];
  cudaLaunchConfig_t cfg = cluster_config(D, at, s);
  cfg.numAttrs = use_pdl() ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, cluster_kernel(D), D, x, b, c0_first ? 1 : 0);
  if (e != cudaSuccess) {
    set_error(std::string("cluster launch: ") + cudaGetErrorString(e));
    return GMG_ERR_CUDA;
  }
  GMG_LAUNCHED();
  return GMG_OK;
}
template gmg_status launch_cluster<float>(gmg_ctx*, float*, const float*, bool, cudaStream_t);
template gmg_status launch_cluster<double>(gmg_ctx*, double*, const double*, bool, cudaStream_t);

// The polls after which the waits of this handle's cluster launches give up.
void set_wait_polls(gmg_ctx* c, int polls) {
  c->wait_polls = polls;
  c->cl32.polls = c->cl64.polls = polls < 0 ? kWaitPolls : polls;
}

// Self-test of the bounded wait: one warp waits on an mbarrier that nothing
// arrives on, so every poll fails and the wait gives up; elapsed device time
// in *ns.
__global__ void k_wait_selftest(int polls, int* err, unsigned long long* ns) {
  __shared__ uint64_t bar;
  const uint32_t m = smem_addr(&bar);
  if (threadIdx.x == 0) mbar_init(m, 1);
  __syncthreads();
  unsigned long long t0, t1;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  mbar_wait(m, 0u, err, polls);
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t1));
  if (threadIdx.x == 0) *ns = t1 - t0;
}

// GMG_ERR_TIMEOUT once if a wait of a cluster launch gave up (its results are
// then not to be trusted); clears the flag.
gmg_status cluster_status(gmg_ctx* c, cudaStream_t s) {
  int* err = c->cl32.l0 >= 0 ? c->cl32.err : c->cl64.l0 >= 0 ? c->cl64.err : nullptr;
  if (!err) return GMG_OK;
  int h = 0;
  GMG_CK(cudaMemcpyAsync(&h, err, sizeof(int), cudaMemcpyDeviceToHost, s));
  GMG_CK(cudaStreamSynchronize(s));
  if (h) {
    GMG_CK(cudaMemsetAsync(err, 0, sizeof(int), s));
    set_error("cluster launch: a wait for tables, matrix entries or another CTA's values timed out");
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
