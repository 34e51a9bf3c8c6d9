// Internal structures of libgmg (not part of the ABI).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cstdint>
#include <cstdlib>
#include <memory>
#include <string>
#include <utility>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "gmg.h"
#include "gmg_fpbits.cuh"

namespace gmg {

constexpr int kSlice = 32;          // rows per sliced-ELL slice (one warp)
constexpr int kHashSlots = 1024;    // per-warp hash table of the Galerkin product
constexpr int kMaxRowEntries = 768; // Galerkin row limit (3/4 of the table)
constexpr int64_t kMaxCoarse = 8192;
constexpr int kRedBlocks = 608;     // fixed grid of the deterministic reductions (4 x 152 SMs)
constexpr int kMaxRhs = 16;
// Index of a multi-right-hand-side block width NR (1, 2, 4, 8, 16) in per-width tables.
constexpr int nr_index(int NR) { return NR == 1 ? 0 : NR == 2 ? 1 : NR == 4 ? 2 : NR == 8 ? 3 : 4; }

void set_error(const std::string& msg);

// Kernels launched by this library on the calling thread (graph replays add
// the number of kernel nodes captured in the graph).
extern thread_local uint64_t g_launches;

#define GMG_LAUNCHED()                                                                    \
  do {                                                                                    \
    ++::gmg::g_launches;                                                                  \
    cudaError_t e_ = cudaGetLastError();                                                  \
    if (e_ != cudaSuccess) {                                                              \
      ::gmg::set_error(std::string("kernel launch: ") + cudaGetErrorString(e_));          \
      return GMG_ERR_CUDA;                                                                \
    }                                                                                     \
  } while (0)

#define GMG_CK(call)                                                                      \
  do {                                                                                    \
    cudaError_t e_ = (call);                                                              \
    if (e_ != cudaSuccess) {                                                              \
      ::gmg::set_error(std::string(#call) + ": " + cudaGetErrorString(e_));               \
      return e_ == cudaErrorMemoryAllocation ? GMG_ERR_OOM : GMG_ERR_CUDA;                \
    }                                                                                     \
  } while (0)

#define GMG_TRY(call)                     \
  do {                                    \
    gmg_status s_ = (call);               \
    if (s_ != GMG_OK) return s_;          \
  } while (0)

// Programmatic dependent launch: a kernel may start while its predecessor
// drains; `pdl_wait` blocks until the predecessor grid has completed and its
// writes are visible, `pdl_trigger` lets the successor start launching.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// GMG_NO_PDL=1 turns programmatic dependent launch off (plain stream order);
// g_pdl_suspended turns it off for the launches of the calling thread.
extern thread_local bool g_pdl_suspended;
inline bool use_pdl() {
  static const bool on = [] {
    const char* e = std::getenv("GMG_NO_PDL");
    return !(e && e[0] == '1');
  }();
  return on && !g_pdl_suspended;
}

// Launches `k` on `s` with programmatic stream serialisation.
template <typename... P, typename... A>
inline gmg_status launch(void (*k)(P...), int64_t grid, int block, cudaStream_t s, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::max<int64_t>(1, grid));
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = use_pdl() ? 1 : 0;
  cudaError_t e = cudaLaunchKernelEx(&cfg, k, std::forward<A>(args)...);
  ++g_launches;
  if (e != cudaSuccess) {
    set_error(std::string("kernel launch: ") + cudaGetErrorString(e));
    return GMG_ERR_CUDA;
  }
  return GMG_OK;
}

// Device allocation registry of a handle: everything is freed by gmg_destroy.
// A named range on the host timeline of a profiler (NVTX; next to no cost
// when no tool is attached).  next() ends the current range and opens another.
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  void next(const char* name) {
    nvtxRangePop();
    nvtxRangePushA(name);
  }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

struct Arena {
  std::vector<void*> ptrs;
  double ms_alloc = 0.0, ms_copy = 0.0;  // host time in cudaMalloc and in uploads (GMG_VERBOSE=1 reports it)
  int64_t n_alloc = 0;
  template <class T>
  gmg_status alloc(T** p, size_t n) {
    *p = nullptr;
    if (n == 0) n = 1;
    const auto t0 = std::chrono::steady_clock::now();
    cudaError_t e = cudaMalloc((void**)p, n * sizeof(T));
    ms_alloc += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
    ++n_alloc;
    if (e != cudaSuccess) {
      cudaGetLastError();  // reported here, not by the next launch
      set_error(std::string("cudaMalloc: ") + cudaGetErrorString(e));
      return GMG_ERR_OOM;
    }
    ptrs.push_back(*p);
    return GMG_OK;
  }
  void release() {
    for (void* p : ptrs) cudaFree(p);
    ptrs.clear();
  }
  void release_one(void* p) {
    for (auto& q : ptrs)
      if (q == p) {
        cudaFree(q);
        q = ptrs.back();
        ptrs.pop_back();
        return;
      }
  }
};

// Set-up tables are copied (and cleared) through the legacy stream from pageable
// memory: such a call may return while the last of it is on its way, and a
// caller's stream need not wait for that stream.  Called before the first
// kernel that reads them.
inline gmg_status uploads_landed() {
  GMG_CK(cudaStreamSynchronize(cudaStreamLegacy));
  return GMG_OK;
}

// A sliced-ELL matrix: rows grouped in slices of 32 consecutive rows; slice s
// stores width_s columns as [k][lane] (entry (row0_s + lane, k) at
// ptr[s] + k * 32 + lane), so a warp's loads of one k are contiguous.
// Padding entries carry weight 0 and a valid column.
struct Ell {
  int64_t nslice = 0, entries = 0;
  int64_t* ptr = nullptr;     // nslice + 1 entry offsets
  int32_t* row0 = nullptr;    // first row of each slice
  int32_t* nrow = nullptr;    // rows in each slice (<= 32)
  int32_t* col = nullptr;
  double* v64 = nullptr;
  float* v32 = nullptr;
};

struct Level {
  int64_t n = 0, nnz = 0;
  int ncolor = 0;
  int lanes = 1;   // warps sharing one row in Gauss-Seidel (1, 2, 4, 8)
  int mlanes[5] = {0, 0, 0, 0, 0};  // the same for the multi-right-hand-side kernels, by block width
                                    // NR = 1, 2, 4, 8, 16 (0: default by mean row length)
  int rlanes = 1;  // the same for the residual (all rows at once, so more parallel)
  std::vector<int64_t> color_off;        // host: first permuted row of each colour (+ end)
  std::vector<int64_t> color_slice_off;  // host: first slice of each colour (+ end)
  std::vector<int32_t> h_color;          // host: colour of every row (caller numbering)
  std::vector<int32_t> h_key;            // host: locality rank of every row (caller numbering)
  std::vector<int64_t> h_ptr;            // host: entry offsets of the slices of A (set-up only)
  // numbering: perm[new] = old, iperm[old] = new
  int32_t* perm = nullptr;
  int32_t* iperm = nullptr;
  // Galerkin operator in caller numbering (CSR, FP64): source of all values
  int64_t* csr_rowptr = nullptr;
  int32_t* csr_col = nullptr;
  double* csr_val = nullptr;
  int64_t* csr2ell = nullptr;  // ELL slot of each CSR entry, or -1 - row for the diagonal (levels > 0)
  // Galerkin plan of this level (l > 0): terms of entry e are
  // plan_edge/plan_coef[plan_ptr[e] .. plan_ptr[e+1]) (CSR positions in level
  // l-1 and P_iJ P_jK), in canonical order; empty below the diagonal
  int64_t* plan_ptr = nullptr;
  int32_t* plan_edge = nullptr;
  double* plan_coef = nullptr;
  int64_t plan_terms = 0;
  // the same plan sliced for the numeric pass (entries with terms, sorted by
  // term count, 32 per slice, terms stored [k][lane], zero-padded)
  int64_t plan_nup = 0;
  int64_t plan_long_slices = 0;  // leading slices whose width exceeds 32 terms
  int32_t* plan_up = nullptr;
  int32_t* plan_mirror = nullptr;  // CSR position of each entry's mirror, -1 on the diagonal
  int64_t* plan_sptr = nullptr;
  int32_t* plan_sedge = nullptr;
  double* plan_scoef = nullptr;
  // off-diagonal part of A_l in the permuted numbering
  Ell A;
  double* diag64 = nullptr;
  double* dinv64 = nullptr;
  float* diag32 = nullptr;
  float* dinv32 = nullptr;
  // prolongation P_l to the next level, caller numbering (Galerkin product input)
  int64_t nc = 0;
  int32_t* p_idx_o = nullptr;
  double* p_w_o = nullptr;
  int64_t* pt_rowptr_o = nullptr;  // columns of P_l (caller numbering)
  int32_t* pt_col_o = nullptr;
  double* pt_w_o = nullptr;
  // prolongation in the permuted numbering of both levels
  int32_t* p_idx = nullptr;
  double* p_w64 = nullptr;
  float* p_w32 = nullptr;
  // restriction P_l^T as sliced ELL over the next level's permuted rows
  Ell R;
  // work vectors (permuted numbering); batched forms use nrhs columns
  double *x64 = nullptr, *b64 = nullptr, *r64 = nullptr;
  float *x32 = nullptr, *b32 = nullptr, *r32 = nullptr;
  float *X32 = nullptr, *B32 = nullptr, *R32 = nullptr;  // [n x kMaxRhs]
};

// The coarse part of a V-cycle on one thread-block cluster (gmg_cluster.cu):
// the smoothed levels l0 .. lambda-1 and the coarsest, rows split over the
// CTAs.  Offsets are bytes into the dynamic shared memory of every CTA (the
// same layout in each); images are per CTA in global memory, copied whole.
constexpr int kClMaxLevels = 6;         // smoothed levels in the cluster
constexpr int kClStages = 4;            // entry buffers (the current phase and up to three ahead)
constexpr int kSmemLimit = 227 * 1024;  // the largest dynamic shared memory of a CTA (no static shared memory)
template <class T>
struct ClusterLevel {
  int ncolor, tpr, lg_tpr, r_tpr, lg_r_tpr;  // lanes per row of the sweeps and of the restriction from this level
  bool streamed;                             // entries stream from L2 instead of staying in shared memory
  int n_own_max, n_loc_max, rsl_max, r_max;
  // shared memory: the image (header, halo bytes of the transfers' phases,
  // slices, colour records or the coarsest level's global rows, halo stores of
  // x and of the residual; level l0: partners, stream steps), the values
  // (pairs of b and 1/a_ii, a_ii, then resident entry units), x (own and halo
  // rows).  Header: own rows, own and halo rows,
  // slices, restriction slices, own rows of colour 0, halo stores [5], [6) of
  // the rows that the post-smoothing updates first, partners, own rows of the
  // coarsest level, halo stores of x, of its colour 0, of the residual
  int o_img, o_val, o_x;
  int img_bytes, val_bytes;
  int i_ex, i_sl, i_cr, i_xd, i_rd, v_diag, v_ent;
  const char *img, *vimg;
  const uint16_t* p_idx;  // per CTA 3 x n_own_max: the prolongation into this level
  const T* p_w;
  const int4* r_sl;       // per CTA rsl_max slices of the restriction from this level, r_max terms
  const uint16_t* r_col;
  const T* r_w;
  const int32_t *vsrc, *dsrc;  // where the entries and the diagonal come from (refresh)
  int64_t nvsrc, n_ent, n_stream;  // entries of all CTAs, of a CTA, streamed
};
template <class T>
struct ClusterDesc {
  int l0 = -1;  // first level (-1: no cluster)
  int ncta = 0, nlev = 0, nc = 0;
  int nu_pre = 0, nu_post = 0, post_forward = 0;
  bool coarse64 = false;  // FP32 cycles: coarsest solve with the FP64 inverse and FP64 sums
  int nstage = 0, nsteps = 0, stage_bytes = 0;
  int o_mbar = 0, o_tok = 0, o_r[2] = {0, 0}, o_bc = 0, o_bd = 0, o_buf = 0, i_steps = 0, i_partners = 0, smem = 0;
  int* err = nullptr;  // set when a bounded wait gave up (for a table, an entry block or a message)
  int polls = 0;       // limit of each wait
  const T* ainv = nullptr;
  const double* ainv64 = nullptr;
  const int32_t* l2g = nullptr;  // level l0: global rows of each CTA's own and halo rows
  const uint4* s_ent = nullptr;  // streamed entry units
  const int32_t* s_src = nullptr;
  ClusterLevel<T> lv[kClMaxLevels + 1] = {};
  bool wide[kClMaxLevels] = {};  // one thread per row (the per-colour kernels' sums)
};

}  // namespace gmg

struct gmg_ctx {
  gmg_options opt{};
  int device = 0;
  int nlev = 0;
  double p_unity_dev = 0.0;  // largest |sum_k w_ik - 1| over the rows of every P_l
  std::vector<gmg::Level> L;
  gmg::Arena arena;
  // coarsest level
  int64_t nco = 0;
  double* dense = nullptr;  // npad x npad sweep work matrix (npad = n rounded up to 32)
  double* Ainv = nullptr;   // A_lambda^-1 (symmetric, full, n x n)
  double* dbuf = nullptr;   // two 32 x 32 pivot inverses, panel U and U D^-1 (npad x 32 each)
  int* gj_cnt = nullptr;    // per sweep: arrival counter of the next pivot tile, then work counter
  int nsm = 1;              // SMs of the device (persistent grids)
  // A(t) = M + t L kept split (gmg_setup_ML): lumped mass, L values (caller
  // CSR order), position of every row's diagonal entry
  double* ml_M = nullptr;
  double* ml_L = nullptr;
  int64_t* ml_dpos = nullptr;
  double ml_t = 0.0;
  // cycles run levels >= cl32.l0 (FP32) or cl64.l0 (FP64) as one cluster launch
  bool single_rhs = true;  // false: a member of a many-mesh handle, whose cycles are all batched
  gmg::ClusterDesc<float> cl32{};
  gmg::ClusterDesc<double> cl64{};
  // handles whose solves run FP64 cycles: the FP32 tables are built for the first
  // FP32 cycle, and filled again for the first one after a refresh (by every
  // refresh once a caller's capture holds an FP32 cycle that reads them as they are)
  bool cl32_late = false, cl32_stale = false, cl32_captured = false;
  bool cl_off = false, cl_small = false;  // GMG_NO_TAIL, GMG_NO_CLUSTER_LEVEL and
  int cl_ctas = 0;                        // GMG_TAIL_CTAS at set-up (0: 16, else 8)
  int wait_polls = -1;                    // limit of the cluster launches' waits (-1: the default)
  float* Ainv32 = nullptr;  // coarsest inverse in FP32 for the cluster launch
  int* dstatus = nullptr;   // device status words
  // outer iteration (finest level, permuted numbering, FP64)
  double *xs = nullptr, *bs = nullptr, *rs = nullptr, *zs = nullptr, *ps = nullptr, *qs = nullptr, *ros = nullptr;
  double* io = nullptr;    // n x kMaxRhs staging for caller-numbered vectors
  double* io2 = nullptr;
  double* XS = nullptr;    // batched FP64 iterate [n x kMaxRhs]
  double* RS = nullptr;    // batched FP64 residual
  double* BS = nullptr;
  double* red = nullptr;   // reduction partials
  int64_t red_cap = 0;     // capacity of `red` in doubles
  int* red_cnt = nullptr;  // arrival counters of the fused last-block reductions (zero between launches)
  double* scal = nullptr;  // device scalars (norms, dots)
  double* h_scal = nullptr;  // pinned host mirror
  // captured iteration bodies, indexed by mode * 2 + segment
  cudaGraphExec_t graphs[8] = {};
  uint64_t graph_kernels[8] = {};  // kernel nodes of each captured graph
  // device-driven solves per mode: graphs whose conditional WHILE node repeats
  // the iteration until the convergence test fails on the device.  [mode][1]
  // starts at the initial residual; [mode][0] (CG only) after the start's
  // cycle, for a start that ran on the stream
  cudaGraphExec_t loops[4][2] = {};
  uint64_t loop_once[4][2] = {};     // kernel nodes outside the loop
  uint64_t loop_kernels[4] = {};     // kernel nodes of one loop iteration
  bool loop_refused[4][2] = {};      // instantiation failed: the host loop serves what this graph would
  // the same for the batched solve, by block width NR = 1, 2, 4, 8, 16
  cudaGraphExec_t mloops[5] = {};
  uint64_t mloop_kernels[5] = {};
  bool mloop_refused[5] = {};
  int* dloop = nullptr;           // device iteration counter, iteration limit, columns
  double* dhist = nullptr;        // relative residual per iteration (max_iter + 1)
  cudaStream_t g_stream = nullptr;
  bool values_ready = false;
  // the coarsest inverse of a numeric refresh runs on its own stream while the
  // caller's next work starts; ev_inv marks its end, and until a call joins it
  // (inv_pending) nothing may read the inverse; its pivot check is read at the
  // join (inv_check)
  cudaStream_t inv_stream = nullptr;
  cudaEvent_t ev_gal = nullptr, ev_inv = nullptr;
  bool inv_pending = false, inv_check = false;
  // kernel timing: events bracket the finest level's smoothing blocks
  // (0-1 pre, 2-3 post) and the whole cycle (4-5)
  bool prof = false;
  bool prof_pending = false;
  cudaEvent_t ev[6] = {};
  double prof_acc[4] = {0, 0, 0, 0};  // smoothing ms, GS launches, cycle ms, cycles
  int prof_gs = 0;                    // finest-level GS launches of the last timed cycle
  // per-level timing of the same cycles: six events per level (before and
  // after pre-smoothing, after the restriction, after the coarser levels,
  // after the prolongation, after post-smoothing); levels run inside the
  // cluster launch or as the coarsest solve record only the first and last
  std::vector<cudaEvent_t> lev_ev;
  std::vector<int> lev_kind;    // per level: 0 not recorded, 1 all six events, 2 first and last only
  std::vector<int> lev_gs;      // GS launches of the level in the last timed cycle
  std::vector<double> lev_acc;  // per level: smoothing ms, GS launches, transfer ms, whole-level ms
};

namespace gmg {
// Makes `s` wait for a coarsest inverse still running on its own stream; with
// `check` also reads its pivot check (host synchronisation).
gmg_status join_inverse(gmg_ctx* c, cudaStream_t s, bool check);
// Reads the pivot check of a joined inverse once (GMG_ERR_CHOLESKY on failure).
gmg_status inverse_status(gmg_ctx* c, cudaStream_t s);
// The cluster form of the coarse levels (gmg_cluster.cu): tables from the
// levels' patterns and numberings, for the precision of the handle's cycles
// (built on host threads between start and finish, which uploads them; the
// arguments outlive the job), values after a numeric set-up, the launch x <- MGI(x, b, l0), and the state of its bounded
// waits.
struct ClusterJob;
std::shared_ptr<ClusterJob> start_cluster(gmg_ctx* c, const std::vector<std::vector<int64_t>>& hrp,
                                          const std::vector<std::vector<int32_t>>& hcol,
                                          const std::vector<std::vector<int32_t>>& perm,
                                          const std::vector<std::vector<int32_t>>& iperm, const gmg_prolong* P);
gmg_status finish_cluster(gmg_ctx* c, ClusterJob& job);
// The FP32 tables of a handle whose solves run FP64 cycles, if they have not
// been built; with `values` also filled from the level values.  Nothing is
// built while s is capturing (the cycle then runs as launches per colour).
gmg_status late_cluster(gmg_ctx* c, cudaStream_t s, bool values);
gmg_status refresh_cluster_values(gmg_ctx* c, cudaStream_t s);
template <class T>
gmg_status launch_cluster(gmg_ctx* c, T* x, const T* b, bool c0_first, cudaStream_t s);
gmg_status cluster_status(gmg_ctx* c, cudaStream_t s);
void set_wait_polls(gmg_ctx* c, int polls);
}  // namespace gmg
