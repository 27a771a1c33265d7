// Zalesak flux-corrected transport passes (Sec. 2.1): the explicit FE-SSP stage
// (Sec. 2.1.2) and the Crank-Nicolson residual (Sec. 2.1.1), both with Zalesak's
// limiter (Sec. 2.1.3).
//
// Structure.  Each pass of a stage is one kernel over the rows; a pair's flux
// r_ij is computed once, by the row of its lower node, and stored in r_up (the
// upper half of the pattern, r_ji = -r_ij).  The node passes that need all
// fluxes of a row (P+/-, then alpha and F*) read r_up at their own row and,
// shifted by the column offset, at the rows of their lower neighbours.  On
// GB300 the FP64 pipe, not HBM, bounds these passes, so each pair costs as few
// FP64 operations as the formulas allow and every comparison, min and max runs
// on the integer pipe (kernels_common.cuh).
#include "afc_internal.h"
#include "grid_sync.cuh"
#include "kernels_common.cuh"
#include "ssp_rows.cuh"

namespace afc {

namespace {

// ---- explicit stage (per-row arithmetic in ssp_rows.cuh) ------------------------

// On grids of at most kPdlRows rows consecutive passes of a step are launched with
// programmatic dependent launch: a pass lets the next one launch once all its blocks run,
// and waits for the one before it (which has waited for its own predecessor) before it
// touches anything a pass writes.  On larger grids the waiting blocks take the place of
// running ones (SSP3 step in double, us, with / without: P1 9^3 62 / 68, Q1 17^3 81 / 86, Q1 25^3
// 84 / 86, Q1 33^3 113 / 90, Q1 41^3 179 / 117).  With graph = 1 these sizes take the one-launch step
// (k_ssp_step) instead, so that this serves host-driven steps.
constexpr int64_t kPdlRows = 16384;
constexpr int64_t kStepRows = 16384;   // the graph form's one-launch step (k_ssp_step)

template <int KT, bool MIXED>
__global__ void k_ssp_rate(Offsets of, SspArrays a, const double* __restrict__ u, double dt) {
  pdl_trigger();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (i < a.N) ssp_rate_row<KT, MIXED>(of, a, i, u, dt);
}

template <int KT, bool MIXED>
__global__ void k_ssp_edges(Offsets of, SspArrays a, const double* __restrict__ u) {
  pdl_trigger();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (i < a.N) ssp_edges_row<KT, MIXED>(of, a, i, u);
}

template <int KT, bool MIXED, bool SMALL, bool FUSED>
__global__ void k_ssp_factors(Offsets of, SspArrays a, const double* u, double dt) {
  pdl_trigger();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (i < a.N) ssp_factors_row<KT, MIXED, FUSED, kGroup<KT>, SMALL>(of, a, i, u, dt);
}

template <int KT, bool MIXED, bool SMALL>
__global__ void k_ssp_correct(Offsets of, SspArrays a, int limiter, double dt, double ca,
                              const double* uA, double cb, double* out) {
  pdl_trigger();
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  pdl_wait();
  if (i < a.N) ssp_correct_row<KT, MIXED, kGroup<KT>, SMALL>(of, a, i, limiter, dt, ca, uA, cb, out);
}
// Below this many rows the passes take their SMALL form: one resident wave of it (Q1 at 89 to 96
// registers: two blocks of 256 on each of 152 SMs); beyond that its registers cost more than its
// loads in flight gain.  SSP3 step, us, large / small form: Q1 mixed 68,921 rows 115 / 105, 91,125 130 / 133,
// 274,625 249 / 303; Q1 in double 35,937 rows 95.2 / 94.7, 91,125 154 / 160; P1 in double 1 % of each
// other up to 117,649.  The mixed form takes 56 to 72 registers for the other patterns: P1 117,649 rows
// 108 / 101, 274,625 166 / 165, 389,017 223 / 229.
constexpr int64_t kSmallRows = 2 * 152 * kBlock, kSmallRowsMixed = 300000;
// In the mixed mode their factors pass is FUSED: a flux is three FP32 operations, a launch costs
// more (77,121 rows of Q1: 114 us a step against 119 us).  Not in double (P1 9^3: 67 us against 61 us),
// and not on larger grids or in batches (48 mixed instances: 7.2 ms against 7.0 ms).

// A whole SSP2 / SSP3 step of a small problem as one cooperative launch, its passes separated
// by grid barriers: on grids of a few thousand rows a pass is latency (one to two microseconds),
// and a launch costs more than a barrier of as many blocks (SSP3 step in double, us, against
// launches with programmatic dependent launch: P1 9^3 56 / 60, P1 25^3 62 / 70, Q1 17^3 72 / 81, Q1 25^3 75 / 84;
// mixed Q1 17^3 84 / 91).
constexpr int kStepBlock = 128;

struct StepVecs {
  double *u, *v, *w;   // u^n and the result; stage vectors
};

template <int KT, bool MIXED>
__global__ void __launch_bounds__(kStepBlock) k_ssp_step(Offsets of, SspArrays a, StepVecs x, int stages, int limiter,
                                                         double dt, GridBar* bar, unsigned long long wait_ns,
                                                         long long* key, double* h) {
  const int64_t i = blockIdx.x * (int64_t)kStepBlock + threadIdx.x;
  const bool row = i < a.N;
  constexpr int S = kGroup<KT>;
  for (int st = 0; st < stages; ++st) {
    const bool last = st == stages - 1;
    const double* in = st == 0 ? x.u : st == 1 ? x.v : x.w;
    double* out = last ? x.u : st == 0 ? x.v : x.w;
    const double ca = st == 0 ? 0.0 : stages == 2 ? 0.5 : st == 1 ? 0.75 : 1.0 / 3.0;
    const double cb = st == 0 ? 1.0 : stages == 2 ? 0.5 : st == 1 ? 0.25 : 2.0 / 3.0;
    if (row) ssp_rate_row<KT, MIXED>(of, a, i, in, dt);
    grid_barrier(bar, wait_ns);
    if (limiter != AFC_LIM_NONE && !(MIXED && limiter == AFC_LIM_ZALESAK)) {
      if (row) ssp_edges_row<KT, MIXED>(of, a, i, in);
      grid_barrier(bar, wait_ns);
    }
    if (limiter == AFC_LIM_ZALESAK) {
      if (row) ssp_factors_row<KT, MIXED, MIXED, S, true>(of, a, i, in, dt);
      grid_barrier(bar, wait_ns);
    }
    if (row) ssp_correct_row<KT, MIXED, S, true>(of, a, i, limiter, dt, ca, x.u, cb, out);
    if (!last) grid_barrier(bar, wait_ns);
  }
  Range r;
  if (row) r.add(x.u[i]);   // this thread's own store
  if (r.finish(key, h)) h[62] = (double)*(volatile int*)&bar->err;
}

// (m_ij, d_ij) of the pairs in single precision
__global__ void k_pairs_to_float(int64_t n, const double* __restrict__ m, const double* __restrict__ d,
                                 float2* __restrict__ md) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) md[i] = make_float2(__double2float_rn(m[i]), __double2float_rn(d[i]));
}

// ---- Crank-Nicolson -------------------------------------------------------------

// Once per step: y = AA u_old, predictor u~ = u_old - (dt/2)(y - f)/m (Eq. forward_euler,
// u_D at Dirichlet nodes), b0 = (m/dt) u_old - y/2 + f (right-hand side of Eq. CNZal).
template <int KT>
__global__ void k_cn_predictor(int64_t N, Offsets of, const double* __restrict__ AA, const double* __restrict__ uo,
                               const double* __restrict__ f, const double* __restrict__ mL,
                               const uint8_t* __restrict__ dir, const double* __restrict__ udir, double dt,
                               double* __restrict__ ut, double* __restrict__ b0) {
  const int K = KT > 0 ? KT : of.K;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  double y = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) y = fma(AA[k * N + i], uo[i + of.o[k]], y);
  const double m = mL[i];
  ut[i] = dir[i] ? udir[i] : uo[i] - 0.5 * dt * (y - f[i]) / m;
  b0[i] = (m / dt * uo[i] - 0.5 * y) + f[i];
}

// m_i Q+/- of the CN predictor over N_i (fixed for the whole step, so the product
// with the lumped mass is formed once per step rather than in every factors pass).
template <int KT>
__global__ void k_bounds_of(int64_t N, Offsets of, const unsigned long long* __restrict__ mask,
                            const double* __restrict__ v, const double* __restrict__ mL, double* __restrict__ Qp,
                            double* __restrict__ Qm) {
  const int K = KT > 0 ? KT : of.K;
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const unsigned long long mk = mask[i];
  const double vi = v[i];
  long long kmax = dkey(vi), kmin = kmax;
#pragma unroll
  for (int k = 0; k < K; ++k) {
    if (!((mk >> k) & 1ull)) continue;
    const long long kj = dkey(v[i + of.o[k]]);
    kmax = kj > kmax ? kj : kmax;
    kmin = kj < kmin ? kj : kmin;
  }
  const double m = mL[i];
  Qp[i] = m * (from_key(kmax) - vi);
  Qm[i] = m * (from_key(kmin) - vi);
}

// Node sums of the CN flux: a = u - u_old, s = u + u_old (at the start of a step; each
// solve renews them in its last pass).
__global__ void k_cn_update(int64_t N, const double* __restrict__ u, const double* __restrict__ uo,
                            double* __restrict__ a, double* __restrict__ s) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double ui = u[i], uoi = uo[i];
  a[i] = ui - uoi;
  s[i] = ui + uoi;
}

// Eq. flux_002 for every pair i < j, prelimited by Eq. prelimiting (L = 2) against twice
// its diffusive part at the CN average:  q = d_ij (s_j - s_i) = 2 d_ij (ubar_j - ubar_i),
// r = (m_ij / dt)(a_i - a_j) + q / 2,  r <- minmod(r, q).
// One thread per pair slot: block = 32 rows (threadIdx.x) x all upper offsets (threadIdx.y).
template <int KT>
__global__ void k_cn_edges(int64_t N, Offsets of, const double* __restrict__ mdt_up, const double* __restrict__ d_up,
                           const double* __restrict__ a, const double* __restrict__ s, int prelimit,
                           double* __restrict__ r_up) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  const int ku = threadIdx.y;
  const int64_t i = blockIdx.x * (int64_t)32 + threadIdx.x;
  if (i >= N) return;
  const int64_t q = (int64_t)ku * N + i;
  const int64_t j = i + of.o[Kup + 1 + ku];
  pdl_trigger();
  const double dq = d_up[q], mq = mdt_up[q];   // no pass of the step writes them
  pdl_wait();
  const double lim = dq * (s[j] - s[i]);
  double r = fma(mq, a[i] - a[j], half_exact(lim));
  if (prelimit) r = minmod(r, lim);
  r_up[q] = r;
}

// Zalesak steps 1-3 for the CN fluxes (Q+/- precomputed from the predictor).
template <int KT>
__global__ void k_cn_factors(int64_t N, Offsets of, const unsigned long long* __restrict__ mask,
                             const double* __restrict__ r_up, const double* __restrict__ mQp,
                             const double* __restrict__ mQm,
                             const uint8_t* __restrict__ dir, double dt, double* __restrict__ Rp,
                             double* __restrict__ Rm) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  pdl_trigger();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  // the mask, the Dirichlet flag and m Q+/- (formed once per step) before the wait for
  // the fluxes of the edge pass
  const bool isdir = dir[i];
  const unsigned long long mk = mask[i];
  const double qp = mQp[i], qm = mQm[i];
  pdl_wait();
  if (isdir) { Rp[i] = 1.0; Rm[i] = 1.0; return; }
  SignedSums128 acc;
  constexpr int S = kGroup<KT>;
#pragma unroll
  for (int k0 = 0; k0 < K; k0 += S) {
    double r[S];
#pragma unroll
    for (int j = 0; j < S; ++j)
      if (k0 + j != Kup) r[j] = r_up[pair_slot(of, Kup, group_at<KT>(k0 + j, K), i, N)];
#pragma unroll
    for (int j = 0; j < S; ++j) {
      const int k = k0 + j;
      if (k == Kup || !((mk >> k) & 1ull)) continue;
      acc.add((unsigned long long)__double_as_longlong(r[j]) ^ (k > Kup ? 0ull : 0x8000000000000000ull));
    }
  }
  double Pp, Pm;
  acc.result(Pp, Pm);
  Rp[i] = zalesak_factor(qp, dt * Pp);
  Rm[i] = zalesak_factor(qm, dt * Pm);
}

// Zalesak step 4, F*, and the nonlinear residual of Eq. CNZal:
// res = b0 + F* - (m/dt u + AA u / 2) on free rows, 0 on Dirichlet rows;
// block partial sums of res^2 for the stopping test.  (The system matrix M_L/dt + AA/2 in place
// of AA saves 0.6 % of a step at Q1 65^3, one matrix less in L2, but its rounded diagonal shows in
// the result: 6.7e-16 against 5.7e-16 from the step in 64 bits.)
template <int KT>
__global__ void __launch_bounds__(256, 4) k_cn_residual(int64_t N, Offsets of, int limiter, const unsigned long long* __restrict__ mask,
                              const double* __restrict__ r_up, const double* __restrict__ AA,
                              const double* __restrict__ un, const double* __restrict__ Rp,
                              const double* __restrict__ Rm,
                              const double* __restrict__ b0,
                              const double* __restrict__ mLdt, const uint8_t* __restrict__ dir,
                              double* __restrict__ res, double* __restrict__ Fout, double* __restrict__ part) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  pdl_trigger();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double r2 = 0.0;
  // y = AA u from the matrix and the state, before the wait for the factors pass: no pass
  // of the limiter writes them (u is the solver's, complete before the edge pass started)
  const bool act = i < N && !dir[i];
  double y = 0.0;
  if (act) {
#pragma unroll
    for (int k = 0; k < K; ++k) y = fma(AA[k * N + i], un[i + of.o[k]], y);
  }
  pdl_wait();
  if (i < N) {
    double rv = 0.0, F = 0.0;
    if (act) {
      const unsigned long long mk = mask[i];
      if (limiter != AFC_LIM_NONE) {
        const double rpi = Rp[i], rmi = Rm[i];
        constexpr int S = kGroup<KT>;
#pragma unroll
        for (int k0 = 0; k0 < K; k0 += S) {
          double r[S], Rj[S];
#pragma unroll
          for (int j = 0; j < S; ++j) {
            if (k0 + j == Kup) continue;
            r[j] = r_up[pair_slot(of, Kup, group_at<KT>(k0 + j, K), i, N)];
            if (k0 + j < Kup) r[j] = neg_bits(r[j]);
          }
          if (limiter == AFC_LIM_ZALESAK) {   // R- of the neighbour for r > 0, R+ else: one load each
#pragma unroll
            for (int j = 0; j < S; ++j)
              if (k0 + j != Kup) Rj[j] = (gt0(r[j]) ? Rm : Rp)[i + of.o[group_at<KT>(k0 + j, K)]];
          }
#pragma unroll
          for (int j = 0; j < S; ++j) {
            const int k = k0 + j;
            if (k == Kup || !((mk >> k) & 1ull)) continue;
            if (limiter == AFC_LIM_ZALESAK) F = fma(imin_nn(gt0(r[j]) ? rpi : rmi, Rj[j]), r[j], F);
            else F += r[j];
          }
        }
      }
      rv = b0[i] + F - (mLdt[i] * un[i] + 0.5 * y);
    }
    res[i] = rv;
    if (Fout) Fout[i] = F;
    r2 = rv * rv;
  }
  block_sum_to(r2, part);
}

}  // namespace

SspArrays ssp_arrays(afc_problem_s* p) {
  SspArrays a;
  a.N = p->N;
  a.AA = p->AA.p;
  a.m_up = p->m_up.p;
  a.d_up = p->d_up.p;
  a.md32 = p->md32.p;
  a.mL = p->mL.p;
  a.imL = p->imL.p;
  a.f = p->f.p;
  a.dir = p->dir.p;
  a.udir = p->udir.p;
  a.mask = p->mask.p;
  a.udot = p->udot.p;
  a.ut = p->ut.p;
  a.uw = p->uw.p;
  a.r_up = p->r_up.p;
  a.r32 = p->r32.p;
  a.Rp = p->Rp.p;
  a.Rm = p->Rm.p;
  a.Fs = p->Fs.p;
  return a;
}

int ensure_ssp_mixed(afc_problem_s* p) {
  if (p->ssp32_ready) return AFC_OK;
  const int64_t N = p->N, Kup = p->Kup;
  int st;
  if ((st = p->md32.alloc(Kup * N)) || (st = p->r32.alloc(Kup * N)) || (st = p->uw.alloc(N, p->pad))) return st;
  AFC_LAUNCH(p, "k_pairs_to_float", k_pairs_to_float<<<grid_for(Kup * N), kBlock, 0, p->stream>>>(
                                        Kup * N, p->m_up.p, p->d_up.p, p->md32.p));
  AFC_CUDA(cudaGetLastError());
  p->ssp32_ready = true;
  return AFC_OK;
}

int fe_stage(afc_problem_s* p, const double* uin, double dt, int limiter, double a, const double* uA, double b,
             double* out, bool mixed, bool pdl) {
  const int64_t N = p->N;
  const dim3 g((unsigned)grid_for(N)), blk(kBlock);
  cudaStream_t s = p->stream;
  if (mixed) {
    int st = ensure_ssp_mixed(p);
    if (st) return st;
  }
  const SspArrays arr = ssp_arrays(p);
  const bool chain = N <= kPdlRows;
  pdl = pdl && chain;
  if (limiter == AFC_LIM_MC) {
    // transient MC (Sec. 2.2): rate, clipped fluxes, then the unweighted sum of r*
    int st = AFC_OK;
    with_K(p->K, [&](auto kc) {
      constexpr int KT = decltype(kc)::value;
      AFC_LAUNCH(p, "k_ssp_rate", launch_pass(false, k_ssp_rate<KT, false>, g, blk, s, p->offs, arr, uin, dt));
      if ((st = mc_ssp_fluxes(p, uin))) return;
      AFC_LAUNCH(p, "k_ssp_correct", launch_pass(false, k_ssp_correct<KT, false, false>, g, blk, s, p->offs, arr,
                                                 (int)AFC_LIM_GALERKIN, dt, a, uA, b, out));
    });
    if (st) return st;
    AFC_CUDA(cudaGetLastError());
    return AFC_OK;
  }
  auto run = [&](auto kc, auto mc) {
    constexpr int KT = decltype(kc)::value;
    constexpr bool MX = decltype(mc)::value;
    AFC_LAUNCH(p, "k_ssp_rate", launch_pass(pdl, k_ssp_rate<KT, MX>, g, blk, s, p->offs, arr, uin, dt));
    const bool small = N < (MX && KT != 27 ? kSmallRowsMixed : kSmallRows);
    const bool fused = MX && small && limiter == AFC_LIM_ZALESAK;
    if (limiter != AFC_LIM_NONE && !fused)
      AFC_LAUNCH(p, "k_ssp_edges", launch_pass(chain, k_ssp_edges<KT, MX>, g, blk, s, p->offs, arr, uin));
    auto factors = small ? k_ssp_factors<KT, MX, true, MX> : k_ssp_factors<KT, MX, false, false>;
    if (limiter == AFC_LIM_ZALESAK)
      AFC_LAUNCH(p, "k_ssp_factors", launch_pass(chain, factors, g, blk, s, p->offs, arr, uin, dt));
    auto correct = small ? k_ssp_correct<KT, MX, true> : k_ssp_correct<KT, MX, false>;
    AFC_LAUNCH(p, "k_ssp_correct", launch_pass(chain, correct, g, blk, s, p->offs, arr, limiter, dt, a, uA, b, out));
  };
  with_K(p->K, [&](auto kc) {
    if (mixed) run(kc, std::true_type{});
    else run(kc, std::false_type{});
  });
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

int ssp_stages(afc_problem_s* p, const afc_opts* o) {
  const bool mixed = o->precision == AFC_MIXED;
  const int lim = o->limiter;
  const double dt = o->dt;
  double *u = p->u.p, *v = p->ustage.p, *w = p->tmp.p;
  // u^n stays in u until the last stage, whose passes read it at their own row only, in the
  // pass that writes it
  int st = fe_stage(p, u, dt, lim, 0.0, nullptr, 1.0, v, mixed);
  if (st) return st;
  if (o->scheme == AFC_SSP2) return fe_stage(p, v, dt, lim, 0.5, u, 0.5, u, mixed, true);
  if ((st = fe_stage(p, v, dt, lim, 0.75, u, 0.25, w, mixed, true))) return st;
  return fe_stage(p, w, dt, lim, 1.0 / 3.0, u, 2.0 / 3.0, u, mixed, true);
}

bool ssp_one_launch(const afc_problem_s* p, const afc_opts* o) {
  return p->N <= kStepRows && o->limiter != AFC_LIM_MC;
}

int ssp_step_launch(afc_problem_s* p, const afc_opts* o) {
  const SspArrays arr = ssp_arrays(p);
  const StepVecs x{p->u.p, p->ustage.p, p->tmp.p};
  cudaError_t e = cudaSuccess;
  auto run = [&](auto kc, auto mc) {
    constexpr int KT = decltype(kc)::value;
    constexpr bool MX = decltype(mc)::value;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid_for(p->N, kStepBlock));
    cfg.blockDim = dim3(kStepBlock);
    cfg.stream = p->stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    AFC_LAUNCH(p, "k_ssp_step",
               e = cudaLaunchKernelEx(&cfg, k_ssp_step<KT, MX>, p->offs, arr, x, o->scheme == AFC_SSP2 ? 2 : 3,
                                      (int)o->limiter, o->dt, reinterpret_cast<GridBar*>(p->bar.p),
                                      kBarrierWaitNs, p->range.p, p->host_scal));
  };
  with_K(p->K, [&](auto kc) {
    if (o->precision == AFC_MIXED) run(kc, std::true_type{});
    else run(kc, std::false_type{});
  });
  if (e != cudaSuccess) return cuda_fail(e, "cudaLaunchKernelEx(k_ssp_step)");
  return AFC_OK;
}

namespace {
// linear Zal+CN: u = 2 u~ - u_old (the value u^n is replaced by in Eq. flux_002), u_D on Dirichlet rows
__global__ void k_cn_linear_guess(int64_t N, const uint8_t* __restrict__ dir, const double* __restrict__ udir,
                                  const double* __restrict__ ut, const double* __restrict__ u_old,
                                  double* __restrict__ u) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < N) u[i] = dir[i] ? udir[i] : 2.0 * ut[i] - u_old[i];
}
}  // namespace

int cn_linear_guess(afc_problem_s* p, const double* u_old, double* u) {
  AFC_LAUNCH(p, "k_cn_linear_guess", k_cn_linear_guess<<<grid_for(p->N), kBlock, 0, p->stream>>>(
                                         p->N, p->dir.p, p->udir.p, p->ut.p, u_old, u));
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

int cn_predictor(afc_problem_s* p, const double* u_old, double dt) {
  const int64_t N = p->N;
  const int64_t g = grid_for(N);
  cudaStream_t s = p->stream;
  with_K(p->K, [&](auto kc) {
    constexpr int KT = decltype(kc)::value;
    AFC_LAUNCH(p, "k_cn_predictor", k_cn_predictor<KT><<<g, kBlock, 0, s>>>(N, p->offs, p->AA.p, u_old, p->f.p,
                                                                             p->mL.p, p->dir.p, p->udir.p, dt, p->ut.p,
                                                                             p->b0.p));
    AFC_LAUNCH(p, "k_bounds_of",
               k_bounds_of<KT><<<g, kBlock, 0, s>>>(N, p->offs, p->mask.p, p->ut.p, p->mL.p, p->Qp.p,
                                                    p->Qm.p));
  });
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

int cn_update(afc_problem_s* p, const double* u, const double* u_old) {
  AFC_LAUNCH(p, "k_cn_update",
             k_cn_update<<<grid_for(p->N), kBlock, 0, p->stream>>>(p->N, u, u_old, p->cn_a.p, p->cn_s.p));
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

namespace {

// F*_i = sum_j r*_ij of the clipped fluxes stored once per pair (0 on Dirichlet rows)
template <int KT>
__global__ void k_pair_sum(int64_t N, Offsets of, const unsigned long long* __restrict__ mask,
                           const double* __restrict__ r_up, const uint8_t* __restrict__ dir, double* __restrict__ F) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  double s = 0.0;
  if (!dir[i]) {
    const unsigned long long mk = mask[i];
#pragma unroll
    for (int k = 0; k < K; ++k) {
      if (k == Kup || !((mk >> k) & 1ull)) continue;
      s += pair_flux(of, Kup, k, i, N, r_up);
    }
  }
  F[i] = s;
}

// res = b0 + (F*(u) + Fold) / 2 - (m/dt u + AA u / 2) on free rows, block partials of res^2
template <int KT>
__global__ void __launch_bounds__(256, 3) k_mccn_residual(
    int64_t N, Offsets of, const unsigned long long* __restrict__ mask, const double* __restrict__ r_up,
    const double* __restrict__ AA, const double* __restrict__ u, const double* __restrict__ Fold,
    const double* __restrict__ b0, const double* __restrict__ mLdt, const uint8_t* __restrict__ dir,
    double* __restrict__ res, double* __restrict__ Fout, double* __restrict__ part) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  double r2 = 0.0;
  if (i < N) {
    double rv = 0.0, F = 0.0;
    if (!dir[i]) {
      const unsigned long long mk = mask[i];
      double y = 0.0;
#pragma unroll
      for (int k = 0; k < K; ++k) y = fma(AA[k * N + i], u[i + of.o[k]], y);
#pragma unroll
      for (int k = 0; k < K; ++k) {
        if (k == Kup || !((mk >> k) & 1ull)) continue;
        F += pair_flux(of, Kup, k, i, N, r_up);
      }
      F = 0.5 * (F + Fold[i]);
      rv = b0[i] + F - (mLdt[i] * u[i] + 0.5 * y);
    }
    res[i] = rv;
    if (Fout) Fout[i] = F;
    r2 = rv * rv;
  }
  block_sum_to(r2, part);
}

}  // namespace

int mc_cn_old_flux(afc_problem_s* p, const double* u_old) {
  const int64_t N = p->N, g = grid_for(N);
  cudaStream_t s = p->stream;
  const SspArrays arr = ssp_arrays(p);
  int st = AFC_OK;
  with_K(p->K, [&](auto kc) {
    constexpr int KT = decltype(kc)::value;
    AFC_LAUNCH(p, "k_ssp_rate", k_ssp_rate<KT, false><<<g, kBlock, 0, s>>>(p->offs, arr, u_old, 0.0));
    if ((st = mc_ssp_fluxes(p, u_old))) return;
    AFC_LAUNCH(p, "k_pair_sum", k_pair_sum<KT><<<g, kBlock, 0, s>>>(N, p->offs, p->mask.p, p->r_up.p, p->dir.p,
                                                                      p->Fold.p));
  });
  if (st) return st;
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

int mc_cn_residual(afc_problem_s* p, const double* u, double* res, double* normsq_slot) {
  const int64_t N = p->N, g = grid_for(N);
  cudaStream_t s = p->stream;
  const SspArrays arr = ssp_arrays(p);
  int st = AFC_OK;
  with_K(p->K, [&](auto kc) {
    constexpr int KT = decltype(kc)::value;
    AFC_LAUNCH(p, "k_ssp_rate", k_ssp_rate<KT, false><<<g, kBlock, 0, s>>>(p->offs, arr, u, 0.0));
    if ((st = mc_ssp_fluxes(p, u))) return;
    AFC_LAUNCH(p, "k_mccn_residual",
               k_mccn_residual<KT><<<g, kBlock, 0, s>>>(N, p->offs, p->mask.p, p->r_up.p, p->AA.p, u, p->Fold.p,
                                                        p->b0.p, p->mLdt.p, p->dir.p, res, p->Fs.p, p->part.p));
  });
  if (st) return st;
  if (normsq_slot) finalize_sum(p, p->part.p, (int)g, normsq_slot);
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

int cn_limited_residual(afc_problem_s* p, const double* u_new, double dt, int limiter, int prelimit, double* res,
                        double* normsq_slot) {
  const int64_t N = p->N;
  const int64_t g = grid_for(N);
  cudaStream_t s = p->stream;
  with_K(p->K, [&](auto kc) {
    constexpr int KT = decltype(kc)::value;
    if (limiter != AFC_LIM_NONE)
      AFC_LAUNCH(p, "k_cn_edges", k_cn_edges<KT><<<grid_for(N, 32), dim3(32, p->Kup), 0, s>>>(N, p->offs, p->mdt_up.p, p->d_up.p, p->cn_a.p,
                                                                       p->cn_s.p, prelimit, p->r_up.p));
    // programmatic dependent launch down the limiter passes (the edge pass follows the
    // solver with a plain dependency)
    if (limiter == AFC_LIM_ZALESAK)
      AFC_LAUNCH(p, "k_cn_factors", launch_pass(limiter != AFC_LIM_NONE, k_cn_factors<KT>, dim3((unsigned)g),
                                                dim3(kBlock), s, N, p->offs, (const unsigned long long*)p->mask.p,
                                                (const double*)p->r_up.p, (const double*)p->Qp.p,
                                                (const double*)p->Qm.p, (const uint8_t*)p->dir.p, dt, p->Rp.p, p->Rm.p));
    AFC_LAUNCH(p, "k_cn_residual",
               launch_pass(limiter != AFC_LIM_NONE, k_cn_residual<KT>, dim3((unsigned)g), dim3(kBlock), s, N,
                           p->offs, limiter, (const unsigned long long*)p->mask.p, (const double*)p->r_up.p,
                           (const double*)p->AA.p, u_new, (const double*)p->Rp.p, (const double*)p->Rm.p,
                           (const double*)p->b0.p, (const double*)p->mLdt.p, (const uint8_t*)p->dir.p, res, p->Fs.p, p->part.p));
  });
  if (normsq_slot) finalize_sum(p, p->part.p, (int)g, normsq_slot);
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

}  // namespace afc
