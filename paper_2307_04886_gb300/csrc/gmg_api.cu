// extern "C" entry points of libgmg (declared in include/gmg.h).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <exception>
#include <new>
#include <string>
#include <vector>

#include "gmg_cycle.cuh"

namespace gmg {
extern thread_local std::string g_last_error;

static bool is_pcg(int mode) { return mode == GMG_FP32_PCG || mode == GMG_FP64_PCG; }

static gmg_status check_handle(gmg_handle h) {
  if (!h) {
    set_error("null handle");
    return GMG_ERR_INVALID_ARG;
  }
  GMG_CK(cudaSetDevice(h->device));
  return GMG_OK;
}

// Runs one iteration body, from a captured graph when enabled.
static gmg_status run_body(gmg_ctx* c, int mode, int seg, cudaStream_t s) {
  if (!c->opt.use_graphs) return iteration_body(c, mode, seg, s);
  const int key = mode * 2 + seg;
  if (!c->graphs[key]) {
    if (!c->g_stream) GMG_CK(cudaStreamCreateWithFlags(&c->g_stream, cudaStreamNonBlocking));
    cudaGraph_t g = nullptr;
    const uint64_t before = g_launches;
    GMG_CK(cudaStreamBeginCapture(c->g_stream, cudaStreamCaptureModeThreadLocal));
    gmg_status st = iteration_body(c, mode, seg, c->g_stream);
    cudaError_t e = cudaStreamEndCapture(c->g_stream, &g);
    c->graph_kernels[key] = g_launches - before;  // captured, not yet run
    g_launches = before;
    if (st != GMG_OK) {
      if (g) cudaGraphDestroy(g);
      return st;
    }
    GMG_CK(e);
    cudaError_t ei = cudaGraphInstantiate(&c->graphs[key], g, 0);
    cudaGraphDestroy(g);
    GMG_CK(ei);
  }
  GMG_CK(cudaGraphLaunch(c->graphs[key], s));
  g_launches += c->graph_kernels[key];
  return GMG_OK;
}

static gmg_status fetch_scalars(gmg_ctx* c, cudaStream_t s) {
  GMG_CK(cudaMemcpyAsync(c->h_scal, c->scal, 8 * sizeof(double), cudaMemcpyDeviceToHost, s));
  GMG_CK(cudaStreamSynchronize(s));
  if (c->prof && c->prof_pending) {  // the last cycle's events have completed
    float a = 0, b = 0, v = 0;
    GMG_CK(cudaEventElapsedTime(&a, c->ev[0], c->ev[1]));
    GMG_CK(cudaEventElapsedTime(&b, c->ev[2], c->ev[3]));
    GMG_CK(cudaEventElapsedTime(&v, c->ev[4], c->ev[5]));
    c->prof_acc[0] += a + b;
    c->prof_acc[1] += (double)c->prof_gs;
    c->prof_acc[2] += v;
    c->prof_acc[3] += 1;
    for (int l = 0; l < c->nlev && (int)c->lev_ev.size() >= 6 * c->nlev; ++l) {
      cudaEvent_t* E = &c->lev_ev[6 * l];
      double* acc = &c->lev_acc[4 * l];
      float t = 0.f;
      if (c->lev_kind[l] == 1) {
        float p0 = 0, p1 = 0, t0 = 0, t1 = 0;
        GMG_CK(cudaEventElapsedTime(&p0, E[0], E[1]));
        GMG_CK(cudaEventElapsedTime(&p1, E[4], E[5]));
        GMG_CK(cudaEventElapsedTime(&t0, E[1], E[2]));
        GMG_CK(cudaEventElapsedTime(&t1, E[3], E[4]));
        acc[0] += p0 + p1;
        acc[1] += c->lev_gs[l];
        acc[2] += t0 + t1;
      }
      if (c->lev_kind[l] != 0) {
        GMG_CK(cudaEventElapsedTime(&t, E[0], E[5]));
        acc[3] += t;
      }
    }
    c->prof_pending = false;
  }
  return GMG_OK;
}

static gmg_status run_cycle_body(gmg_ctx* c, int mode, int seg, cudaStream_t s) {
  GMG_TRY(run_body(c, mode, seg, s));
  if (c->nlev > 1 && (!is_pcg(mode) || seg == 1)) c->prof_pending = c->prof;
  return GMG_OK;
}

// Destroys every captured graph (their launch shapes or event nodes are stale).
static void drop_graphs(gmg_ctx* c) {
  for (auto& g : c->graphs)
    if (g) {
      cudaGraphExecDestroy(g);
      g = nullptr;
    }
  for (int m = 0; m < 4; ++m) {
    for (auto& g : c->loops[m]) {
      if (g) cudaGraphExecDestroy(g);
      g = nullptr;
    }
    c->loop_refused[m][0] = c->loop_refused[m][1] = false;
  }
}

// Captures what `body` launches on the handle's stream into `g` behind the
// nodes `deps`, which it replaces by the nodes the captured work ends with.
template <class F>
static cudaError_t capture_into(gmg_ctx* c, cudaGraph_t g, std::vector<cudaGraphNode_t>* deps, gmg_status* st,
                                F&& body) {
  cudaError_t e = cudaStreamBeginCaptureToGraph(c->g_stream, g, deps->data(), nullptr, deps->size(),
                                                cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  *st = body();
  cudaStreamCaptureStatus cs;
  const cudaGraphNode_t* tail = nullptr;
  size_t count = 0;
  e = cudaStreamGetCaptureInfo(c->g_stream, &cs, nullptr, nullptr, &tail, nullptr, &count);
  if (e == cudaSuccess && count) deps->assign(tail, tail + count);
  cudaGraph_t done = nullptr;
  const cudaError_t e2 = cudaStreamEndCapture(c->g_stream, &done);
  return e != cudaSuccess ? e : e2;
}

// Builds a device-driven solve of `mode`: the start (with `whole`: the initial
// residual and its test, for CG also the first cycle and direction), for CG the
// first step, a conditional WHILE node (condition 1 at every launch) whose body
// is captured from loop_body, and for CG the true residual at the end.  One
// launch and one synchronisation then serve a solve.  The kernels keep their
// programmatic launch edges if the CUDA driver instantiates them around and
// inside a conditional body, else all is captured again in plain stream order;
// if neither instantiates, the host loop serves what this form would.
static gmg_status build_loop(gmg_ctx* c, int mode, bool whole) {
  if (!c->g_stream) GMG_CK(cudaStreamCreateWithFlags(&c->g_stream, cudaStreamNonBlocking));
  cudaGraphExec_t& exec = c->loops[mode][whole];
  const uint64_t before = g_launches;
  bool pdl = false;
  // a pending coarsest inverse is joined by whoever launches the graph
  const bool pending = c->inv_pending;
  c->inv_pending = false;
  struct Restore {
    gmg_ctx* c;
    bool pending;
    ~Restore() { c->inv_pending = pending; }
  } restore{c, pending};
  for (int attempt = 0; attempt < 2 && !exec; ++attempt) {
    cudaGraph_t g = nullptr;
    GMG_CK(cudaGraphCreate(&g, 0));
    cudaGraphConditionalHandle h = 0;
    std::vector<cudaGraphNode_t> deps, none;
    gmg_status st = GMG_OK;
    uint64_t once = 0;
    g_pdl_suspended = attempt == 1;
    cudaError_t e = cudaGraphConditionalHandleCreate(&h, g, 1, cudaGraphCondAssignDefault);
    if (e == cudaSuccess && (whole || is_pcg(mode)))
      e = capture_into(c, g, &deps, &st, [&]() -> gmg_status {
        if (whole) GMG_TRY(outer_residual_norm(c, true, c->g_stream));
        if (!is_pcg(mode)) return GMG_OK;
        if (whole) GMG_TRY(pcg_start(c, mode, c->g_stream));
        return iteration_body(c, mode, 0, c->g_stream, h, true);
      });
    once = g_launches - before;
    g_launches = before;
    cudaGraphNodeParams np = {};
    if (e == cudaSuccess && st == GMG_OK) {
      np.type = cudaGraphNodeTypeConditional;
      np.conditional.handle = h;
      np.conditional.type = cudaGraphCondTypeWhile;
      np.conditional.size = 1;
      cudaGraphNode_t node;
      e = cudaGraphAddNode(&node, g, deps.data(), nullptr, deps.size(), &np);
      deps.assign(1, node);
    }
    if (e == cudaSuccess && st == GMG_OK)
      e = capture_into(c, np.conditional.phGraph_out[0], &none, &st,
                       [&] { return loop_body(c, mode, h, c->g_stream); });
    c->loop_kernels[mode] = g_launches - before;
    g_launches = before;
    if (e == cudaSuccess && st == GMG_OK && is_pcg(mode)) {
      g_pdl_suspended = true;  // the loop node is no programmatic predecessor
      e = capture_into(c, g, &deps, &st, [&] { return outer_residual_norm(c, false, c->g_stream); });
      once += g_launches - before;
      g_launches = before;
    }
    c->loop_once[mode][whole] = once;
    g_pdl_suspended = false;
    if (st == GMG_OK && e == cudaSuccess) e = cudaGraphInstantiate(&exec, g, 0);
    if (st == GMG_OK && e == cudaSuccess) pdl = attempt == 0 && use_pdl();
    cudaGraphDestroy(g);
    if (st != GMG_OK) {
      exec = nullptr;
      return st;
    }
    if (e != cudaSuccess) {
      cudaGetLastError();
      exec = nullptr;
    }
  }
  if (!exec) c->loop_refused[mode][whole] = true;
  if (const char* e = std::getenv("GMG_VERBOSE"))
    if (e[0] == '1')
      std::fprintf(stderr, "gmg: device-side loop for mode %d: %s\n", mode,
                   !exec ? "refused, host loop" : pdl ? "programmatic launches" : "plain stream order");
  return GMG_OK;
}

// Whether a solve in `mode` runs device-driven: graphs on, no per-cycle timing
// (event nodes are not allowed in a conditional body), GMG_NO_DEVICE_LOOP
// unset, an iteration to do, and the graph instantiated.  GMG_NO_RESTART_LOOP=1
// leaves out the form that continues after a start on the stream (tests: the
// host loop then goes on from a restart, as where that graph is refused).
static gmg_status device_loop_ready(gmg_ctx* c, int mode, bool whole, bool* ok) {
  static const bool off = [] {
    const char* e = std::getenv("GMG_NO_DEVICE_LOOP");
    return e && e[0] == '1';
  }();
  *ok = false;
  if (off || !c->opt.use_graphs || c->prof || c->loop_refused[mode][whole] || c->opt.max_iter <= 0) return GMG_OK;
  if (!whole)
    if (const char* e = std::getenv("GMG_NO_RESTART_LOOP"))
      if (e[0] == '1') return GMG_OK;
  if (!c->loops[mode][whole]) GMG_TRY(build_loop(c, mode, whole));
  *ok = c->loops[mode][whole] != nullptr;
  return GMG_OK;
}

// Copies an n-vector in caller numbering (host or device) into the permuted
// device vector `dst` of level l.
static gmg_status load_vec(gmg_ctx* c, int l, const double* src, int mem, double* dst, double* stage,
                           cudaStream_t s) {
  Level& L = c->L[l];
  if (mem == GMG_MEM_HOST) {
    GMG_CK(cudaMemcpyAsync(stage, src, sizeof(double) * (size_t)L.n, cudaMemcpyHostToDevice, s));
    src = stage;
  }
  return launch_gather(L.n, L.perm, src, dst, s);
}

static gmg_status store_vec(gmg_ctx* c, int l, const double* src, double* dst, int mem, double* stage,
                            cudaStream_t s) {
  Level& L = c->L[l];
  if (mem == GMG_MEM_HOST) {
    GMG_TRY(launch_scatter(L.n, L.perm, src, stage, s));
    GMG_CK(cudaMemcpyAsync(dst, stage, sizeof(double) * (size_t)L.n, cudaMemcpyDeviceToHost, s));
    GMG_CK(cudaStreamSynchronize(s));
    return GMG_OK;
  }
  return launch_scatter(L.n, L.perm, src, dst, s);
}

// The outer iteration of one gmg_solve, from the loaded system on.
struct SolveRun {
  gmg_ctx* c;
  cudaStream_t s;
  int mode;
  double tol;
  gmg_solve_info* info;
  int k = 0;
  double rel = 0.0;
  gmg_status st = GMG_ERR_NOT_CONVERGED;
  bool rewrite = false;      // on_device: xs changes after it was stored
  bool wait_failed = false;  // on_device: a bounded wait ran out

  void record(int kk, double v) {
    if (info && info->history && kk < info->history_cap) info->history[kk] = v;
  }

  // The start's test from ||b||^2 and ||r||^2: false ends the solve.
  gmg_status start(double nb, double rr, bool* go) {
    *go = false;
    if (!std::isfinite(nb)) {
      set_error("gmg_solve: non-finite right-hand side");
      st = GMG_ERR_NONFINITE;
    } else if (nb == 0.0) {
      GMG_CK(cudaMemsetAsync(c->xs, 0, sizeof(double) * (size_t)c->L[0].n, s));
      rewrite = true;
      record(0, 0.0);
      st = GMG_OK;
    } else {
      rel = std::sqrt(rr) / nb;
      record(0, rel);
      if (!std::isfinite(rel)) {
        set_error("gmg_solve: non-finite initial residual");
        st = GMG_ERR_NONFINITE;
      } else {
        *go = true;
      }
    }
    return GMG_OK;
  }

  // Graph launches only (build_loop): the solution goes out with the report of
  // every launch, so a solve whose first report confirms the tolerance has
  // synchronised once.
  gmg_status on_device(double* x, double* x_dev, size_t bytes, bool whole) {
    const double* R = c->h_scal;
    if (!is_pcg(mode)) GMG_TRY(join_inverse(c, s, false));
    if (!whole) {
      GMG_TRY(outer_residual_norm(c, true, s));
      GMG_TRY(pcg_start(c, mode, s));
    }
    for (;;) {
      GMG_CK(cudaGraphLaunch(c->loops[mode][whole], s));
      GMG_TRY(store_solution(c, x_dev, s));
      if (x != x_dev) GMG_CK(cudaMemcpyAsync(x, x_dev, bytes, cudaMemcpyDeviceToHost, s));
      GMG_CK(cudaStreamSynchronize(s));
      wait_failed |= R[REP_WAIT] != 0.0;
      if (R[REP_PIVOT] == 0.0) c->inv_check = false;  // else read, and reported, by inverse_status
      const double nb = std::sqrt(R[REP_NB2]);
      if (R[REP_OK] != 1.0) {  // the start failed its test: x has not been written
        bool go = false;
        return start(nb, R[REP_HIST] * nb, &go);  // infinite or NaN stays so
      }
      const int k1 = (int)R[REP_ITERS];
      if (k1 <= k || k1 > c->opt.max_iter) {
        set_error("device loop: iteration counter out of range");
        return GMG_ERR_CUDA;
      }
      g_launches += c->loop_once[mode][whole] + (uint64_t)(k1 - k - (is_pcg(mode) ? 1 : 0)) * c->loop_kernels[mode];
      const int from = k == 0 ? 0 : k + 1;
      if (info && info->history && from < info->history_cap) {
        const int last = std::min(k1, info->history_cap - 1);
        if (last < REP_HIST_CAP)
          std::copy(R + REP_HIST + from, R + REP_HIST + last + 1, info->history + from);
        else
          GMG_CK(cudaMemcpy(info->history + from, c->dhist + from, sizeof(double) * (size_t)(last - from + 1),
                            cudaMemcpyDeviceToHost));
      }
      k = k1;
      rel = R[REP_REL];
      if (!std::isfinite(rel)) {
        set_error("gmg_solve: iterate became non-finite");
        st = GMG_ERR_NONFINITE;
        return GMG_OK;
      }
      if (rel <= tol && is_pcg(mode)) {  // confirmed on the true residual
        rel = std::sqrt(R[REP_RR]) / nb;
        record(k, rel);
      }
      if (rel <= tol) {
        st = GMG_OK;
        return GMG_OK;
      }
      if (!is_pcg(mode) || k >= c->opt.max_iter) break;
      bool again = false;
      GMG_TRY(device_loop_ready(c, mode, false, &again));
      GMG_TRY(pcg_start(c, mode, s));  // restart from the current iterate
      if (!again) {  // no graph for what follows a restart
        rewrite = true;
        return host_steps(nb);
      }
      whole = false;
    }
    set_error("gmg_solve: max_iter reached");
    return GMG_OK;
  }

  // One synchronisation per iteration.
  gmg_status on_host() {
    GMG_TRY(outer_residual_norm(c, false, s));
    GMG_TRY(fetch_scalars(c, s));
    const double nb = std::sqrt(c->h_scal[S_NB2]);
    bool go = true;
    GMG_TRY(start(nb, c->h_scal[S_RR], &go));
    if (!go) return GMG_OK;
    if (!is_pcg(mode)) GMG_TRY(join_inverse(c, s, false));
    if (is_pcg(mode)) GMG_TRY(pcg_start(c, mode, s));
    return host_steps(nb);
  }

  // The iterations from k on (CG: after a start or restart).
  gmg_status host_steps(double nb) {
    bool fresh = true;  // CG: no step since the (re)start
    while (k < c->opt.max_iter) {
      if (is_pcg(mode) && !fresh) GMG_TRY(run_cycle_body(c, mode, 1, s));
      GMG_TRY(run_cycle_body(c, mode, 0, s));
      GMG_TRY(fetch_scalars(c, s));
      ++k;
      fresh = false;
      rel = std::sqrt(c->h_scal[S_RR]) / nb;
      if (!std::isfinite(rel)) {
        set_error("gmg_solve: iterate became non-finite");
        st = GMG_ERR_NONFINITE;
        return GMG_OK;
      }
      if (rel <= tol && is_pcg(mode)) {  // confirm on the true residual
        GMG_TRY(outer_residual_norm(c, false, s));
        GMG_TRY(fetch_scalars(c, s));
        rel = std::sqrt(c->h_scal[S_RR]) / nb;
        record(k, rel);
        if (rel <= tol) {
          st = GMG_OK;
          return GMG_OK;
        }
        GMG_TRY(pcg_start(c, mode, s));  // restart from the current iterate
        fresh = true;
        continue;
      }
      record(k, rel);
      if (rel <= tol) {
        st = GMG_OK;
        return GMG_OK;
      }
    }
    set_error("gmg_solve: max_iter reached");
    return GMG_OK;
  }
};

}  // namespace gmg

using namespace gmg;

namespace gmg {
gmg_status new_handle(gmg_handle* h, const gmg_csr* A, int n_prolong, const gmg_prolong* P,
                      const int32_t* const* coloring, const gmg_options* opt, bool single_rhs, void* stream) {
  g_last_error.clear();
  if (!h || n_prolong < 0 || (n_prolong > 0 && !P)) {
    set_error("gmg_setup: null output handle or bad prolongation list");
    return GMG_ERR_INVALID_ARG;
  }
  *h = nullptr;
  gmg_ctx* c = new (std::nothrow) gmg_ctx();
  if (!c) return GMG_ERR_OOM;
  c->single_rhs = single_rhs;
  if (opt) c->opt = *opt;
  else gmg_default_options(&c->opt);
  if (const char* e = std::getenv("GMG_NO_GRAPHS"))  // profilers list graph nodes slowly
    if (e[0] == '1') c->opt.use_graphs = 0;
  if (c->opt.nu_pre < 0 || c->opt.nu_post < 0 || c->opt.max_iter < 0 || c->opt.precision < GMG_FP64 ||
      c->opt.precision > GMG_FP64_PCG) {
    set_error("gmg_setup: invalid options");
    delete c;
    return GMG_ERR_INVALID_ARG;
  }
  gmg_status st;
  try {
    st = setup_impl(c, A, n_prolong, P, coloring, (cudaStream_t)stream);
  } catch (const std::exception& e) {  // host memory or threads: no exception leaves a C entry
    set_error(std::string("gmg_setup: ") + e.what());
    st = GMG_ERR_OOM;
  }
  if (st != GMG_OK) {
    std::string keep = g_last_error;
    gmg_destroy(c);
    g_last_error = keep;
    return st;
  }
  *h = c;
  return GMG_OK;
}
}  // namespace gmg

extern "C" {

void gmg_default_options(gmg_options* opt) {
  if (!opt) return;
  opt->precision = GMG_FP32_REFINE;
  opt->nu_pre = 2;
  opt->nu_post = 2;
  opt->max_iter = 100;
  opt->post_forward = 0;
  opt->use_graphs = 1;
}

const char* gmg_status_string(gmg_status s) {
  switch (s) {
    case GMG_OK: return "ok";
    case GMG_ERR_INVALID_ARG: return "invalid argument";
    case GMG_ERR_NOT_SPD: return "matrix not symmetric positive definite";
    case GMG_ERR_EMPTY_P_COLUMN: return "empty prolongation column";
    case GMG_ERR_CHOLESKY: return "coarsest Cholesky factorisation failed";
    case GMG_ERR_NOT_CONVERGED: return "not converged";
    case GMG_ERR_NONFINITE: return "non-finite value";
    case GMG_ERR_OOM: return "out of device memory";
    case GMG_ERR_CUDA: return "CUDA error";
    case GMG_ERR_TIMEOUT: return "device wait timed out";
    case GMG_ERR_TOO_LARGE: return "size limit exceeded";
  }
  return "unknown status";
}

const char* gmg_last_error(void) { return g_last_error.c_str(); }

uint64_t gmg_kernel_launches(void) { return g_launches; }

gmg_status gmg_destroy(gmg_handle h) {
  if (!h) return GMG_OK;
  cudaSetDevice(h->device);
  drop_graphs(h);
  for (auto& g : h->mloops)
    if (g) cudaGraphExecDestroy(g);
  if (h->g_stream) cudaStreamDestroy(h->g_stream);
  for (auto& e : h->ev)
    if (e) cudaEventDestroy(e);
  for (auto& e : h->lev_ev)
    if (e) cudaEventDestroy(e);
  if (h->h_scal) cudaFreeHost(h->h_scal);
  cudaDeviceSynchronize();
  if (h->inv_stream) cudaStreamDestroy(h->inv_stream);
  if (h->ev_gal) cudaEventDestroy(h->ev_gal);
  if (h->ev_inv) cudaEventDestroy(h->ev_inv);
  h->arena.release();
  delete h;
  return GMG_OK;
}

gmg_status gmg_setup(gmg_handle* h, const gmg_csr* A, int n_prolong, const gmg_prolong* P,
                     const int32_t* const* coloring, const gmg_options* opt, void* stream) {
  return new_handle(h, A, n_prolong, P, coloring, opt, true, stream);
}

gmg_status gmg_set_values(gmg_handle h, const double* val, int mem, void* stream) {
  NvtxRange nv("gmg_set_values");
  GMG_TRY(check_handle(h));
  if (!val) {
    set_error("gmg_set_values: null values");
    return GMG_ERR_INVALID_ARG;
  }
  cudaStream_t s = (cudaStream_t)stream;
  Level& L0 = h->L[0];
  GMG_TRY(join_inverse(h, s, false));  // a previous refresh's inverse still reads the level values
  GMG_CK(cudaMemcpyAsync(L0.csr_val, val, sizeof(double) * (size_t)L0.nnz,
                         mem == GMG_MEM_HOST ? cudaMemcpyHostToDevice : cudaMemcpyDeviceToDevice, s));
  return numeric_setup(h, s, true);
}

gmg_status gmg_solve(gmg_handle h, const double* b, double* x, double tol, int mem, gmg_solve_info* info,
                     void* stream) {
  NvtxRange nv("gmg_solve");
  GMG_TRY(check_handle(h));
  if (!b || !x || !(tol >= 0.0) || (mem != GMG_MEM_HOST && mem != GMG_MEM_DEVICE)) {
    set_error("gmg_solve: null vector, negative tolerance or bad memory kind");
    return GMG_ERR_INVALID_ARG;
  }
  gmg_ctx* c = h;
  cudaStream_t s = (cudaStream_t)stream;
  const int64_t n = c->L[0].n;
  const size_t bytes = sizeof(double) * (size_t)n;
  const int mode = c->nlev == 1 ? GMG_FP64 : c->opt.precision;
  const bool host = mem == GMG_MEM_HOST;
  if (host) {
    GMG_CK(cudaMemcpyAsync(c->io, b, bytes, cudaMemcpyHostToDevice, s));
    GMG_CK(cudaMemcpyAsync(c->io2, x, bytes, cudaMemcpyHostToDevice, s));
  }
  GMG_TRY(load_system(c, host ? c->io : b, host ? c->io2 : x, tol, s));
  SolveRun run{c, s, mode, tol, info};
  // a CG start joins a pending coarsest inverse right before its first coarse
  // solve (its down-leg overlaps the inverse), so it runs on the stream, not
  // in a graph; the other modes join before their first iteration, and so does
  // CG where one cluster launch is the whole cycle: there is no down-leg to
  // overlap, and the whole solve is one graph
  if (is_pcg(mode) && (mode == GMG_FP32_PCG ? c->cl32.l0 : c->cl64.l0) == 0) GMG_TRY(join_inverse(c, s, false));
  bool dev = false;
  const bool whole = !(is_pcg(mode) && c->inv_pending);
  GMG_TRY(device_loop_ready(c, mode, whole, &dev));
  if (dev) GMG_TRY(run.on_device(x, host ? c->io2 : x, bytes, whole));
  else GMG_TRY(run.on_host());
  if (!dev || run.rewrite) GMG_TRY(store_vec(c, 0, c->xs, x, mem, c->io2, s));
  if (info) {
    info->iters = run.k;
    info->rel_res = run.rel;
  }
  GMG_TRY(inverse_status(c, s));  // the pivot check of an inverse this solve joined
  if (!dev || run.rewrite || run.wait_failed) GMG_TRY(cluster_status(c, s));
  return run.st;
}

gmg_status gmg_wait_limit(gmg_handle h, int polls) {
  GMG_TRY(check_handle(h));
  set_wait_polls(h, polls);
  drop_graphs(h);  // they hold the limit they were captured with
  return GMG_OK;
}

gmg_status gmg_profile(gmg_handle h, int enable) {
  GMG_TRY(check_handle(h));
  if ((enable != 0) == h->prof) return GMG_OK;
  if (enable && !h->ev[0])
    for (auto& e : h->ev) GMG_CK(cudaEventCreate(&e));
  if (enable && h->lev_ev.empty()) {
    h->lev_ev.assign(6 * h->nlev, nullptr);
    for (auto& e : h->lev_ev) GMG_CK(cudaEventCreate(&e));
    h->lev_kind.assign(h->nlev, 0);
    h->lev_gs.assign(h->nlev, 0);
    h->lev_acc.assign(4 * h->nlev, 0.0);
  }
  drop_graphs(h);  // re-capture with or without the event nodes
  h->prof = enable != 0;
  h->prof_pending = false;
  return GMG_OK;
}

gmg_status gmg_profile_read(gmg_handle h, double* out) {
  if (!h || !out) return GMG_ERR_INVALID_ARG;
  for (int k = 0; k < 4; ++k) {
    out[k] = h->prof_acc[k];
    h->prof_acc[k] = 0.0;
  }
  return GMG_OK;
}

gmg_status gmg_profile_levels(gmg_handle h, double* out) {
  if (!h || !out) return GMG_ERR_INVALID_ARG;
  const bool have = (int)h->lev_acc.size() >= 4 * h->nlev;
  for (int k = 0; k < 4 * h->nlev; ++k) {
    out[k] = have ? h->lev_acc[k] : 0.0;
    if (have) h->lev_acc[k] = 0.0;
  }
  return GMG_OK;
}

// Makes a new warps-per-row choice take effect: captured cycles hold the old
// launch shapes.
static gmg_status apply_lanes(gmg_handle h) {
  drop_graphs(h);
  return GMG_OK;
}

gmg_status gmg_autotune(gmg_handle h, int* lanes_out, void* stream) {
  GMG_TRY(check_handle(h));
  // The sweeps are timed as they run in a solve: captured in a CUDA graph with
  // programmatic launches, where the cost of a phase depends on its CTA count
  // and dependent loads rather than on the host's launch rate.
  GMG_CK(cudaStreamSynchronize((cudaStream_t)stream));
  if (!h->g_stream) GMG_CK(cudaStreamCreateWithFlags(&h->g_stream, cudaStreamNonBlocking));
  cudaStream_t cs = h->g_stream;
  cudaEvent_t e0, e1;
  GMG_CK(cudaEventCreate(&e0));
  GMG_CK(cudaEventCreate(&e1));
  gmg_status st = GMG_OK;
  const uint64_t launches_before = g_launches;
  for (int l = 0; l + 1 < h->nlev && st == GMG_OK; ++l) {
    Level& L = h->L[l];
    const int keep = L.lanes;
    float best_ms = 1e30f;
    int best = keep;
    if (cudaMemsetAsync(L.x32, 0, sizeof(float) * (size_t)L.n, cs) != cudaSuccess ||
        cudaMemsetAsync(L.b32, 0, sizeof(float) * (size_t)L.n, cs) != cudaSuccess) {
      st = GMG_ERR_CUDA;
      break;
    }
    for (int G : {1, 2, 4, 8}) {
      L.lanes = G;
      cudaGraph_t g = nullptr;
      cudaGraphExec_t ge = nullptr;
      if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        st = GMG_ERR_CUDA;
        break;
      }
      for (int sweep = 0; sweep < 4 && st == GMG_OK; ++sweep)
        for (int k = 0; k < L.ncolor && st == GMG_OK; ++k) st = launch_gs_colour<float>(L, k, L.b32, L.x32, cs);
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
        set_error("gmg_autotune: graph capture of the sweeps failed");
        st = GMG_ERR_CUDA;
      }
      if (ge) cudaGraphExecDestroy(ge);
      if (g) cudaGraphDestroy(g);
    }
    L.lanes = st == GMG_OK ? best : keep;
    if (lanes_out) lanes_out[l] = L.lanes;
    // the residual covers every row at once: its own split, timed the same way
    const int rkeep = L.rlanes;
    float rbest_ms = 1e30f;
    int rbest = rkeep;
    for (int G : {1, 2, 4, 8}) {
      if (st != GMG_OK) break;
      L.rlanes = G;
      cudaGraph_t g = nullptr;
      cudaGraphExec_t ge = nullptr;
      if (cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
        st = GMG_ERR_CUDA;
        break;
      }
      for (int rep = 0; rep < 4 && st == GMG_OK; ++rep) st = launch_residual<float>(L, L.x32, L.b32, L.r32, cs);
      const cudaError_t ec = cudaStreamEndCapture(cs, &g);
      if (st == GMG_OK && ec == cudaSuccess && cudaGraphInstantiate(&ge, g, 0) == cudaSuccess) {
        float ms = 0.f;
        cudaGraphLaunch(ge, cs);  // warm-up
        cudaEventRecord(e0, cs);
        for (int rep = 0; rep < 3; ++rep) cudaGraphLaunch(ge, cs);
        cudaEventRecord(e1, cs);
        if (cudaEventSynchronize(e1) != cudaSuccess) st = GMG_ERR_CUDA;
        cudaEventElapsedTime(&ms, e0, e1);
        if (st == GMG_OK && ms < rbest_ms) {
          rbest_ms = ms;
          rbest = G;
        }
      } else if (st == GMG_OK) {
        set_error("gmg_autotune: graph capture of the residuals failed");
        st = GMG_ERR_CUDA;
      }
      if (ge) cudaGraphExecDestroy(ge);
      if (g) cudaGraphDestroy(g);
    }
    L.rlanes = st == GMG_OK ? rbest : rkeep;
  }
  g_launches = launches_before;  // timing launches are not the caller's work
  cudaStreamSynchronize(cs);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st == GMG_OK) st = apply_lanes(h);
  return st;
}

gmg_status gmg_set_lanes(gmg_handle h, const int* lanes) {
  GMG_TRY(check_handle(h));
  if (!lanes) {
    set_error("gmg_set_lanes: null lanes");
    return GMG_ERR_INVALID_ARG;
  }
  for (int l = 0; l + 1 < h->nlev; ++l)
    if (lanes[l] != 1 && lanes[l] != 2 && lanes[l] != 4 && lanes[l] != 8) {
      set_error("gmg_set_lanes: level " + std::to_string(l) + " split " + std::to_string(lanes[l]) +
                " is not 1, 2, 4 or 8");
      return GMG_ERR_INVALID_ARG;
    }
  for (int l = 0; l + 1 < h->nlev; ++l) h->L[l].lanes = h->L[l].rlanes = lanes[l];
  return apply_lanes(h);
}

gmg_status gmg_num_levels(gmg_handle h, int* nlev) {
  if (!h || !nlev) return GMG_ERR_INVALID_ARG;
  *nlev = h->nlev;
  return GMG_OK;
}

gmg_status gmg_warnings(gmg_handle h, uint32_t* flags, double* max_dev) {
  if (!h || !flags) return GMG_ERR_INVALID_ARG;
  *flags = h->p_unity_dev > 1e-12 ? GMG_WARN_P_UNITY : 0u;
  if (max_dev) *max_dev = h->p_unity_dev;
  return GMG_OK;
}

gmg_status gmg_level_info(gmg_handle h, int l, int64_t* n, int64_t* nnz, int* ncolors) {
  if (!h || l < 0 || l >= h->nlev) return GMG_ERR_INVALID_ARG;
  if (n) *n = h->L[l].n;
  if (nnz) *nnz = h->L[l].nnz;
  if (ncolors) *ncolors = h->L[l].ncolor;
  return GMG_OK;
}

gmg_status gmg_level_path(gmg_handle h, int l, int* path) {
  if (!h || !path || l < 0 || l >= h->nlev) return GMG_ERR_INVALID_ARG;
  if (l < h->nlev - 1 && h->cl32_late) {
    GMG_TRY(check_handle(h));
    GMG_TRY(late_cluster(h, nullptr, false));
  }
  if (l == h->nlev - 1)
    *path = 3;
  else if (h->cl32.l0 >= 0 && l >= h->cl32.l0)
    *path = h->cl32.wide[l - h->cl32.l0] ? 1 : 2;
  else
    *path = 0;
  return GMG_OK;
}

gmg_status gmg_level_export(gmg_handle h, int l, int64_t* rowptr, int32_t* col, double* val, int32_t* color) {
  GMG_TRY(check_handle(h));
  if (l < 0 || l >= h->nlev) return GMG_ERR_INVALID_ARG;
  Level& L = h->L[l];
  GMG_CK(cudaDeviceSynchronize());
  if (rowptr) GMG_CK(cudaMemcpy(rowptr, L.csr_rowptr, sizeof(int64_t) * (size_t)(L.n + 1), cudaMemcpyDeviceToHost));
  if (col) GMG_CK(cudaMemcpy(col, L.csr_col, sizeof(int32_t) * (size_t)L.nnz, cudaMemcpyDeviceToHost));
  if (val) GMG_CK(cudaMemcpy(val, L.csr_val, sizeof(double) * (size_t)L.nnz, cudaMemcpyDeviceToHost));
  if (color) std::copy(L.h_color.begin(), L.h_color.end(), color);
  return GMG_OK;
}

// ---- single steps of Alg. 2 (device vectors, caller numbering) ----

static gmg_status to_level(gmg_ctx* c, int l, int fp32, const double* src, double* d64, float* d32,
                           cudaStream_t s) {
  GMG_TRY(launch_gather(c->L[l].n, c->L[l].perm, src, d64, s));
  if (fp32) GMG_TRY(launch_d2f(c->L[l].n, d64, d32, s));
  return GMG_OK;
}
static gmg_status from_level(gmg_ctx* c, int l, int fp32, double* d64, const float* d32, double* dst,
                             cudaStream_t s) {
  if (fp32) GMG_TRY(launch_f2d(c->L[l].n, d32, d64, s));
  return launch_scatter(c->L[l].n, c->L[l].perm, d64, dst, s);
}

gmg_status gmg_smooth(gmg_handle h, int l, int fp32, const double* b, double* x, int nsweep, int descending,
                      void* stream) {
  GMG_TRY(check_handle(h));
  if (l < 0 || l >= h->nlev || !b || !x || nsweep < 0) return GMG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  Level& L = h->L[l];
  GMG_TRY(to_level(h, l, fp32, b, L.b64, L.b32, s));
  GMG_TRY(to_level(h, l, fp32, x, L.x64, L.x32, s));
  for (int it = 0; it < nsweep; ++it)
    for (int q = 0; q < L.ncolor; ++q) {
      const int k = descending ? L.ncolor - 1 - q : q;
      if (fp32) GMG_TRY(launch_gs_colour<float>(L, k, L.b32, L.x32, s));
      else GMG_TRY(launch_gs_colour<double>(L, k, L.b64, L.x64, s));
    }
  return from_level(h, l, fp32, L.x64, L.x32, x, s);
}

gmg_status gmg_residual(gmg_handle h, int l, int fp32, const double* x, const double* b, double* r, void* stream) {
  GMG_TRY(check_handle(h));
  if (l < 0 || l >= h->nlev || !b || !x || !r) return GMG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  Level& L = h->L[l];
  GMG_TRY(to_level(h, l, fp32, b, L.b64, L.b32, s));
  GMG_TRY(to_level(h, l, fp32, x, L.x64, L.x32, s));
  if (fp32) GMG_TRY(launch_residual<float>(L, L.x32, L.b32, L.r32, s));
  else GMG_TRY(launch_residual<double>(L, L.x64, L.b64, L.r64, s));
  return from_level(h, l, fp32, L.r64, L.r32, r, s);
}

gmg_status gmg_restrict(gmg_handle h, int l, int fp32, const double* r, double* bc, void* stream) {
  GMG_TRY(check_handle(h));
  if (l < 0 || l + 1 >= h->nlev || !r || !bc) return GMG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  Level& L = h->L[l];
  Level& C = h->L[l + 1];
  GMG_TRY(to_level(h, l, fp32, r, L.r64, L.r32, s));
  if (fp32) GMG_TRY(launch_restrict<float>(L, L.r32, C.b32, C.x32, s));
  else GMG_TRY(launch_restrict<double>(L, L.r64, C.b64, C.x64, s));
  return from_level(h, l + 1, fp32, C.b64, C.b32, bc, s);
}

gmg_status gmg_prolong_add(gmg_handle h, int l, int fp32, const double* u, double* x, void* stream) {
  GMG_TRY(check_handle(h));
  if (l < 0 || l + 1 >= h->nlev || !u || !x) return GMG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  Level& L = h->L[l];
  Level& C = h->L[l + 1];
  GMG_TRY(to_level(h, l + 1, fp32, u, C.x64, C.x32, s));
  GMG_TRY(to_level(h, l, fp32, x, L.x64, L.x32, s));
  if (fp32) GMG_TRY(launch_prolong<float>(L, C.x32, L.x32, s));
  else GMG_TRY(launch_prolong<double>(L, C.x64, L.x64, s));
  return from_level(h, l, fp32, L.x64, L.x32, x, s);
}

gmg_status gmg_coarse_solve(gmg_handle h, int fp32, const double* b, double* x, void* stream) {
  GMG_TRY(check_handle(h));
  if (!b || !x) return GMG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  GMG_TRY(join_inverse(h, s, true));
  const int l = h->nlev - 1;
  Level& C = h->L[l];
  GMG_TRY(to_level(h, l, fp32, b, C.b64, C.b32, s));
  if (fp32) GMG_TRY(launch_coarse<float>(h, C.b32, C.x32, s));
  else GMG_TRY(launch_coarse<double>(h, C.b64, C.x64, s));
  return from_level(h, l, fp32, C.x64, C.x32, x, s);
}

gmg_status gmg_vcycle(gmg_handle h, int fp32, const double* b, double* x, void* stream) {
  GMG_TRY(check_handle(h));
  if (!b || !x) return GMG_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  GMG_TRY(join_inverse(h, s, true));
  Level& L = h->L[0];
  if (fp32) GMG_TRY(late_cluster(h, s, true));
  // the error word is this cycle's only where a cluster launch is part of it
  const bool cluster = (fp32 ? h->cl32.l0 : h->cl64.l0) >= 0;
  if (cluster) GMG_CK(cudaMemsetAsync(h->dstatus + 3, 0, sizeof(int), s));
  GMG_TRY(to_level(h, 0, fp32, b, L.b64, L.b32, s));
  GMG_TRY(to_level(h, 0, fp32, x, L.x64, L.x32, s));
  if (fp32) GMG_TRY(vcycle<float>(h, 0, s));
  else GMG_TRY(vcycle<double>(h, 0, s));
  if (fp32) GMG_TRY(launch_f2d(L.n, L.x32, L.x64, s));
  return cluster ? launch_scatter_cycle(h, L.x64, x, s) : launch_scatter(L.n, L.perm, L.x64, x, s);
}

}  // extern "C"
