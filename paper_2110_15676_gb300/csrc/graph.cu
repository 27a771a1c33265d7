// One time step or one stationary solve as a single CUDA graph launch.
//
// The damped fixed point of Sec. 4 is a while node: its body evaluates the
// limited residual, and the persistent solver launch that follows first decides
// whether to stop (Eq. tol_formula, the iteration limit, or a fixed count), then
// solves and updates.  The host launches the graph and synchronises once;
// no scalar travels to the host inside the step.  The explicit SSP step is a
// plain captured graph.  Graphs are built on first use and rebuilt when the
// options or the problem's buffers change.
#include <cmath>
#include <cstring>
#include <vector>

#include "graph_util.h"
#include "kernels_common.cuh"

namespace afc {

namespace {

__global__ void k_fp_init(double* sc, double thresh, int fixed, int maxit) {
  if (threadIdx.x != 0) return;
  sc[F_CORR] = 0.0;
  sc[F_INNER] = 0.0;
  sc[F_STATUS] = 0.0;
  sc[F_THRESH] = thresh;
  sc[F_FIXED] = (double)fixed;
  sc[F_MAXIT] = (double)maxit;
  sc[F_REVAL] = 0.0;
  sc[F_TIMEOUT] = 0.0;
}

__global__ void k_copy(int64_t n, const double* __restrict__ x, double* __restrict__ y) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) y[i] = x[i];
}

__global__ void k_apply_dirichlet_g(int64_t N, const uint8_t* __restrict__ dir, const double* __restrict__ udir,
                                    double* __restrict__ u) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < N && dir[i]) u[i] = udir[i];
}

}  // namespace

// Cached executable graph and the kernel count of each of its sections (for the
// launch accounting of afc_profile_read).
struct StepGraph {
  cudaGraphExec_t exec = nullptr;
  std::vector<unsigned char> key;
  int64_t k_pro = 0, k_first = 0, k_outer = 0, k_epi = 0;
  int kind = 0;   // 1 fixed point, 2 explicit SSP
  int unroll = 1; // corrections per turn of the while node
};

namespace {

// Corrections per turn of the while node.  A turn costs about 5 us beside its kernels (P1 49^3
// mixed, 942 corrections: 115.8 ms at one correction a turn, 114.0 at two, 112.6 at four); what
// follows the stop in the same turn finds the status set and returns, but its residual has been
// formed in vain.  So four for stationary solves, which take hundreds of corrections, and one for a
// CN step's dozen (Q1 65^3: 8.23 ms at one, 8.37 at four).  A loop of several begins with a residual
// and a solve of its own: a solve that starts converged stops there (P1 129^3, mixed: 0.28 ms, 0.90 with four residuals).
int unroll_of(int system) { return system == 0 ? 4 : 1; }

std::vector<unsigned char> make_key(afc_problem_s* p, const afc_opts* o, int what) {
  std::vector<unsigned char> k(sizeof(afc_opts) + 64);
  std::memcpy(k.data(), o, sizeof(afc_opts));
  double cdt = p->cn_dt;
  uintptr_t cdt_bits;
  std::memcpy(&cdt_bits, &cdt, sizeof(cdt_bits));
  uintptr_t extra[7] = {(uintptr_t)what, (uintptr_t)p->stream, (uintptr_t)krylov_key(p), (uintptr_t)p->AA.p,
                        (uintptr_t)p->Bcn.p, cdt_bits, (uintptr_t)p->grid_wait_ns};
  std::memcpy(k.data() + sizeof(afc_opts), extra, sizeof(extra));
  return k;
}

void drop(StepGraph*& g) {
  if (!g) return;
  if (g->exec) cudaGraphExecDestroy(g->exec);
  delete g;
  g = nullptr;
}

struct ProfOff {   // no event records inside captured graphs; captured launches are not executions
  afc_problem_s* p;
  bool was = false;
  int64_t launches = 0;
  explicit ProfOff(afc_problem_s* p_) : p(p_), launches(p_->launches) { was = prof_set_enabled(p, false); }
  ~ProfOff() {
    prof_set_enabled(p, was);
    p->launches = launches;
  }
};

// Build the fixed-point graph: prologue, while(outer){ residual; solve }, epilogue (with several
// corrections per turn, the first residual and solve before the loop).  The persistent solve decides
// first whether the loop goes on, and applies and counts the update.
template <class Pro, class Res>
int build_fixed_point(afc_problem_s* p, const afc_opts* o, int system, Pro prologue, Res residual, StepGraph& sg,
                      KrylovEpilogue epi) {
  if (!p->cap_stream) AFC_CUDA(cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking));
  cudaStream_t cs = p->cap_stream;
  ProfOff po(p);
  cudaGraph_t g = nullptr;
  AFC_CUDA(cudaGraphCreate(&g, 0));
  int st = AFC_OK;
  std::vector<cudaGraphNode_t> fr;
  cudaGraphConditionalHandle h_loop;
  const double thresh = std::sqrt((double)p->N) * o->fp_tol;
  auto count = [&](auto&& f) {
    const int64_t l0 = p->launches;
    int s = f();
    return std::make_pair(s, p->launches - l0);
  };
  do {
    auto r1 = count([&]() -> int {
      return capture_into(p, cs, g, fr, [&]() -> int {
        AFC_LAUNCH(p, "k_fp_init", k_fp_init<<<1, 32, 0, p->stream>>>(p->scal.p, thresh, o->fp_fixed_its,
                                                                       o->fp_maxit));
        return prologue();
      }, fr);
    });
    if ((st = r1.first)) break;
    sg.k_pro = r1.second;
    if (cudaGraphConditionalHandleCreate(&h_loop, g, 1, cudaGraphCondAssignDefault) != cudaSuccess) {
      st = cuda_fail(cudaGetLastError(), "cudaGraphConditionalHandleCreate");
      break;
    }
    epi.fp_sc = p->scal.p;
    epi.part = p->part.p;
    epi.npart = (int)grid_for(p->N);
    epi.loop = h_loop;
    sg.unroll = unroll_of(system);
    auto corrections = [&](int n, cudaGraph_t into, std::vector<cudaGraphNode_t>& at) {
      return count([&]() -> int {
        for (int c = 0; c < n; ++c) {
          int s = capture_into(p, cs, into, at, residual, at);
          if (s) return s;
          if ((s = krylov_graph(p, system, o, p->res.p, p->delta.p, cs, into, at, &epi))) return s;
        }
        return AFC_OK;
      });
    };
    if (sg.unroll > 1) {
      auto rf = corrections(1, g, fr);
      if ((st = rf.first)) break;
      sg.k_first = rf.second;
    }
    cudaGraph_t body;
    cudaGraphNode_t loop;
    if ((st = add_conditional(g, fr, h_loop, cudaGraphCondTypeWhile, &body, &loop))) break;
    std::vector<cudaGraphNode_t> bf;
    auto r2 = corrections(sg.unroll, body, bf);
    if ((st = r2.first)) break;
    sg.k_outer = r2.second;
    fr.assign(1, loop);
    auto r4 = count([&]() -> int { return capture_into(p, cs, g, fr, [&]() -> int { return range_device(p, p->u.p); }, fr); });
    if ((st = r4.first)) break;
    sg.k_epi = r4.second;
    cudaGraphExec_t ex = nullptr;
    cudaError_t e = cudaGraphInstantiate(&ex, g, 0);
    if (e != cudaSuccess) { st = cuda_fail(e, "cudaGraphInstantiate"); break; }
    sg.exec = ex;
    sg.kind = 1;
  } while (false);
  cudaGraphDestroy(g);
  return st;
}

int run_fixed_point_graph(afc_problem_s* p, StepGraph& sg, afc_stats* stt) {
  AFC_CUDA(cudaGraphLaunch(sg.exec, p->stream));
  AFC_CUDA(cudaStreamSynchronize(p->stream));
  const double* h = p->host_scal;
  const int64_t reval = (int64_t)h[F_REVAL], corr = (int64_t)h[F_CORR];
  const int64_t looped = sg.k_first ? reval - 1 : reval;   // residuals of the loop
  p->launches += sg.k_pro + sg.k_first + (looped + sg.unroll - 1) / sg.unroll * sg.k_outer + sg.k_epi;
  int status = h[F_STATUS] == 1.0 ? AFC_OK : h[F_STATUS] == 2.0 ? AFC_E_NAN : AFC_NOT_CONVERGED;
  if (h[F_TIMEOUT] != 0.0) {
    // the barrier counter is inconsistent after blocks skipped barriers: clear it so
    // that the next persistent launch starts from a clean state
    const int rs = krylov_reset_barrier(p);
    if (rs) return rs;
    status = AFC_E_TIMEOUT;
    set_error("a grid barrier of the persistent Krylov launch gave up waiting");
  } else if (status == AFC_E_NAN) {
    set_error("non-finite nonlinear residual or Krylov breakdown");
  }
  if (stt) {
    stt->outer_its = (int)corr;
    stt->inner_its = (int)h[F_INNER];
    stt->res0 = h[F_RES0];
    stt->res_final = h[F_RESF];
    stt->umin = h[60];
    stt->umax = h[61];
    stt->status = status;
  }
  return status;
}

}  // namespace

void graph_free(afc_problem_s* p) {
  drop(p->g_step);
  drop(p->g_stat);
  if (p->cap_stream) {
    cudaStreamDestroy(p->cap_stream);
    p->cap_stream = nullptr;
  }
}

int cn_step_graph(afc_problem_s* p, const afc_opts* o, afc_stats* stt) {
  if (const int s0 = krylov_prepare(p, o)) return s0;
  const auto key = make_key(p, o, 1);
  if (!p->g_step || p->g_step->key != key) {
    drop(p->g_step);
    p->g_step = new StepGraph();
    const int lim = o->limiter;
    const double dt = o->dt;
    const KrylovEpilogue epi = step_epilogue(p, o);
    int st = build_fixed_point(
        p, o, 1,
        [&]() -> int {
          const int64_t N = p->N;
          AFC_LAUNCH(p, "k_copy", k_copy<<<grid_for(N), kBlock, 0, p->stream>>>(N, p->u.p, p->u0.p));
          int s = cn_predictor(p, p->u0.p, dt);
          if (s) return s;
          if (lim == AFC_LIM_MC) {
            AFC_LAUNCH(p, "k_apply_dirichlet",
                       k_apply_dirichlet_g<<<grid_for(N), kBlock, 0, p->stream>>>(N, p->dir.p, p->udir.p, p->u.p));
            return mc_cn_old_flux(p, p->u0.p);
          }
          if (o->scheme == AFC_CN_LINEAR) {
            if ((s = cn_linear_guess(p, p->u0.p, p->u.p))) return s;
          } else {
            AFC_LAUNCH(p, "k_apply_dirichlet",
                       k_apply_dirichlet_g<<<grid_for(N), kBlock, 0, p->stream>>>(N, p->dir.p, p->udir.p, p->u.p));
          }
          return cn_update(p, p->u.p, p->u0.p);
        },
        [&]() -> int {
          if (lim == AFC_LIM_MC) return mc_cn_residual(p, p->u.p, p->res.p, nullptr);
          return cn_limited_residual(p, p->u.p, dt, lim, o->prelimit, p->res.p, nullptr);
        },
        *p->g_step, epi);
    if (st) {
      drop(p->g_step);
      return st;
    }
    p->g_step->key = key;
  }
  return run_fixed_point_graph(p, *p->g_step, stt);
}

int stationary_graph(afc_problem_s* p, const afc_opts* o, afc_stats* stt) {
  if (const int s0 = krylov_prepare(p, o)) return s0;
  const auto key = make_key(p, o, 2);
  if (!p->g_stat || p->g_stat->key != key) {
    drop(p->g_stat);
    p->g_stat = new StepGraph();
    const int lim = o->limiter;
    const bool pair = o->precision == AFC_MIXED && (lim == AFC_LIM_MC || lim == AFC_LIM_GALERKIN);
    KrylovEpilogue epi = stationary_epilogue(p, o);
    if (pair) epi.pair = p->up2.p;
    int st = build_fixed_point(
        p, o, 0,
        [&]() -> int {
          AFC_LAUNCH(p, "k_apply_dirichlet", k_apply_dirichlet_g<<<grid_for(p->N), kBlock, 0, p->stream>>>(
                                                 p->N, p->dir.p, p->udir.p, p->u.p));
          AFC_CUDA(cudaGetLastError());
          return pair ? mc_pair_split(p, p->u.p) : AFC_OK;
        },
        [&]() -> int {
          // the state's float pairs come from the prologue, then from each solve's update (5 us of a
          // correction at P1 49^3, 14 us at 129^3, when a pass of the sweep formed them)
          if (pair) return mc_pair_residual(p, p->u.p, lim, p->res.p, nullptr, false);
          return mc_limited_residual(p, p->u.p, lim, p->res.p, nullptr);
        },
        *p->g_stat, epi);
    if (st) {
      drop(p->g_stat);
      return st;
    }
    p->g_stat->key = key;
  }
  return run_fixed_point_graph(p, *p->g_stat, stt);
}

int ssp_step_graph(afc_problem_s* p, const afc_opts* o, afc_stats* stt) {
  const bool mixed = o->precision == AFC_MIXED, one = ssp_one_launch(p, o);
  if (mixed) {
    int s0 = ensure_ssp_mixed(p);   // allocation and conversion stay outside the capture
    if (s0) return s0;
  }
  const auto key = make_key(p, o, 3);
  if (!p->g_step || p->g_step->key != key) {
    drop(p->g_step);
    p->g_step = new StepGraph();
    if (!p->cap_stream) AFC_CUDA(cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking));
    ProfOff po(p);
    cudaGraph_t g = nullptr;
    AFC_CUDA(cudaGraphCreate(&g, 0));
    std::vector<cudaGraphNode_t> fr;
    const int64_t l0 = p->launches;
    int st = capture_into(p, p->cap_stream, g, fr, [&]() -> int {
      if (one) return ssp_step_launch(p, o);
      const int s = ssp_stages(p, o);
      return s ? s : range_device(p, p->u.p);
    }, fr);
    if (!st) {
      cudaGraphExec_t ex = nullptr;
      cudaError_t e = cudaGraphInstantiate(&ex, g, 0);
      if (e != cudaSuccess) st = cuda_fail(e, "cudaGraphInstantiate");
      else p->g_step->exec = ex;
    }
    cudaGraphDestroy(g);
    if (st) {
      drop(p->g_step);
      return st;
    }
    p->g_step->k_pro = p->launches - l0;
    p->g_step->kind = 2;
    p->g_step->key = key;
  }
  AFC_CUDA(cudaGraphLaunch(p->g_step->exec, p->stream));
  AFC_CUDA(cudaStreamSynchronize(p->stream));
  p->launches += p->g_step->k_pro;
  if (one && p->host_scal[62] != 0.0) {   // the barrier's state is inconsistent after blocks skipped it
    AFC_CUDA(cudaMemsetAsync(p->bar.p, 0, 4 * sizeof(unsigned int), p->stream));
    AFC_CUDA(cudaStreamSynchronize(p->stream));
    set_error("a grid barrier of the explicit step's launch gave up waiting");
    return AFC_E_TIMEOUT;
  }
  if (stt) {
    stt->stages = o->scheme == AFC_SSP2 ? 2 : 3;
    stt->umin = p->host_scal[60];
    stt->umax = p->host_scal[61];
    stt->status = AFC_OK;
  }
  return AFC_OK;
}

}  // namespace afc
