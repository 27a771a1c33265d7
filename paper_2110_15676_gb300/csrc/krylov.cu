// Jacobi-preconditioned Krylov solvers for the constant M-matrix systems of the
// fixed-point iteration (Sec. 4; Tables 1 and 3: BiCGStab, GMRES, Jacobi), run
// entirely on the device: a solve is one persistent cooperative launch whose
// phases are separated by bounded grid barriers.  Every block forms the solver
// scalars (rho, alpha, omega, Hessenberg columns, Givens rotations) from the
// same partial sums in the same order, so all blocks branch alike and results do
// not depend on scheduling.
//
// Vector type T is double (FP64) or float (the FP32 inner solve of the mixed
// mode, with FP32 matrix values).  What a thread adds over its rows is in T; everything from there on
// is in double, but for the dots of single-precision GMRES, which are added in single precision in
// a defined order up to 256 values (k_gm_single).
#include <climits>
#include <cmath>
#include <cstring>

#include "afc_internal.h"
#include "graph_util.h"
#include "kernels_common.cuh"
#include "grid_sync.cuh"
#include "pair_float.cuh"

namespace afc {

int64_t grid_for(int64_t n, int block) { return (n + block - 1) / block; }

template <class T>
int DBuf<T>::alloc(int64_t n_, int64_t pad_) {
  pad_ = (pad_ + 31) & ~(int64_t)31;   // the logical start stays on a 128-byte boundary
  if (base && n == n_ && pad == pad_) return AFC_OK;
  free_();
  size_t bytes = (size_t)(n_ + 2 * pad_) * sizeof(T);
  if (bytes == 0) bytes = sizeof(T);
  cudaError_t e = device_alloc((void**)&base, bytes, true);   // zero-filled, ready for any stream
  if (e != cudaSuccess) {
    base = nullptr;
    cudaGetLastError();
    set_error(std::string("device allocation of ") + std::to_string(bytes) + " bytes failed: " + cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? AFC_E_OOM : AFC_E_CUDA;
  }
  n = n_;
  pad = pad_;
  p = base + pad_;
  return AFC_OK;
}

template <class T>
void DBuf<T>::free_() {
  if (base) device_free(base);
  base = p = nullptr;
  n = pad = 0;
}

template struct DBuf<double>;
template struct DBuf<float>;
template struct DBuf<int32_t>;
template struct DBuf<uint8_t>;
template struct DBuf<unsigned long long>;
template struct DBuf<float4>;
template struct DBuf<float2>;
template struct DBuf<long long>;

namespace {

__global__ void k_finalize_sum(const double* __restrict__ part, int n, double* __restrict__ out) {
  const double t = final_sum(part, n);
  if (threadIdx.x == 0) *out = t;
}

}  // namespace

void finalize_sum(afc_problem_s* p, const double* part, int n, double* out) {
  AFC_LAUNCH(p, "k_finalize_sum", k_finalize_sum<<<1, 256, 0, p->stream>>>(part, n, out));
}

// ---------------------------------------------------------------------------
// BLAS-1 helpers on double vectors (outer loop)
// ---------------------------------------------------------------------------
namespace {

__global__ void __launch_bounds__(kBlock) k_range(int64_t N, const double* __restrict__ x, long long* key,
                                                  const double* __restrict__ sc, double* h) {
  Range r;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N; i += (int64_t)gridDim.x * blockDim.x) r.add(x[i]);
  if (r.finish(key, h) && threadIdx.x == 0)
    for (int q = 0; q < 12; ++q) h[q] = sc[q];
}

template <class T, class TV>
__global__ void k_spmv(int64_t N, Offsets of, const T* __restrict__ A, const TV* __restrict__ x, TV* __restrict__ y) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= N) return;
  TV s = 0;
#pragma unroll 4
  for (int k = 0; k < of.K; ++k) s = fma((TV)A[k * N + i], x[i + of.o[k]], s);
  y[i] = s;
}

}  // namespace

int range_device(afc_problem_s* p, const double* x) {
  // at most two blocks per SM: each ends in three atomics on one line
  const int g = (int)std::min<int64_t>(grid_for(p->N, 4 * kBlock), 304);
  AFC_LAUNCH(p, "k_range", k_range<<<g, kBlock, 0, p->stream>>>(p->N, x, p->range.p, p->scal.p, p->host_scal));
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

int minmax_device(afc_problem_s* p, const double* x, double* mn, double* mx) {
  const int st = range_device(p, x);
  if (st) return st;
  AFC_CUDA(cudaStreamSynchronize(p->stream));
  *mn = p->host_scal[60];
  *mx = p->host_scal[61];
  return AFC_OK;
}

int dia_spmv(afc_problem_s* p, const double* A, const double* x, double* y) {
  AFC_LAUNCH(p, "k_spmv", k_spmv<double, double><<<grid_for(p->N), kBlock, 0, p->stream>>>(p->N, p->offs, A, x, y));
  AFC_CUDA(cudaGetLastError());
  return AFC_OK;
}

// ---------------------------------------------------------------------------
// Solver workspace
// ---------------------------------------------------------------------------
constexpr int kMaxRestart = 32;   // GMRES(m), m <= 32: a Hessenberg column has an entry per lane of a warp

// device scalar slots
enum : int {
  S_RHO = 0, S_RHO_OLD, S_ALPHA, S_OMEGA, S_TOL, S_NRES, S_N0, S_ITS, S_DONE, S_MAXIT, S_BETA, S_ATOL, S_RTOL,
  S_CYCLES,   // GMRES restart cycles begun (true-residual evaluations)
  S_BERR,     // persistent launches: a grid barrier gave up waiting
  S_END
};
// S_DONE: 0 running, 1 converged, 2 breakdown / non-finite, 3 converged at s (x update pending), 4 maxit

// A solver flag (a double slot holding 0 or a positive code) tested on its bit pattern:
// a compare of doubles issues on GB300's FP64 pipe, where every warp instruction
// costs 16 cycles, and the kernels below test their flags in every thread.
__device__ __forceinline__ bool flag_set(const double* sc, int slot) {
  return (__double_as_longlong(sc[slot]) << 1) != 0;
}
// float -> double without the FP64 pipe (exact; the FP64 instance passes through)
__device__ __forceinline__ double to_dbl(float x) { return widen_exact(x); }
__device__ __forceinline__ double to_dbl(double x) { return x; }

constexpr size_t kHscBytes = (S_END + 8) * sizeof(double);   // host mirror of the scalars

struct KrylovWork {
  int64_t N = 0;
  int pad = 0, m = 0, fp32 = -1;
  DBuf<char> vec;       // all vectors (with halos)
  DBuf<double> sc, part;
  DBuf<unsigned int> barrier;   // GridBar of the persistent launches
  int nsm = 0;                  // SMs of the device (0: not asked yet)
  double* hsc = nullptr;
  size_t vstride = 0;   // elements per vector incl. halo
};

template struct DBuf<char>;
template struct DBuf<unsigned int>;
template struct DBuf<uint16_t>;

namespace {

// ---- BiCGStab (van der Vorst 1992), Jacobi preconditioner on the directions, as one
// persistent cooperative launch --------------------------------------------------
// The five phases of an iteration (p update, v = B phat, s update, t = B shat, x / r
// update) run in one launch, separated by grid barriers; nothing returns to the
// host or the graph between iterations.  Block b owns the contiguous rows
// [N b / G, N (b + 1) / G), at most one block per SM, as many warps as the rows fill: every
// barrier and grid-wide sum costs more with more blocks, and a block's FP64 sums cost 16
// cycles per warp.
//
// What a block alone reads (r, rhat, p, v, t, x) stays in shared memory where its rows fit
// (FP64: up to 660,000 rows in all); phat and shat, which the products of other blocks gather,
// are in global memory.  The scalars of an iteration are formed by one lane per block (the
// first of warp 0, which also polls the barriers and adds the partials) and handed to the
// block through shared memory: formed by every warp, their divisions and square roots held
// the FP64 pipe for about a microsecond per phase.
//
// Measured on one GB300, a CN solve of 3.5 iterations: Q1 65^3 in double 235 -> 198 us, mixed
// 169 -> 120 us; P1 33^3 in double 107 -> 75 us (vectors in global memory, 512 threads in
// every block, scalars in every warp before).
constexpr int kFusedBlock = 512;
constexpr int kBicgVectors = 8;             // phat, shat and the six local ones
constexpr size_t kFusedSmem = 160 * 1024;   // shared memory for a block's six vectors (the rest stays L1)

template <class T>
struct BicgArgs {
  int64_t N;
  double* sc;
  const double* rhs;
  double* xout;
  T* loc;             // the six vectors in global memory, when not in shared memory
  size_t vstride;
  double* part;
  GridBar* bar;
  double atol, rtol;
  int maxit, rows;
  KrylovEpilogue ep;
  unsigned long long wait_ns;
};

template <class T>
struct BicgShared {
  double col[2][kFusedBlock], quarter[2][4];
  double rho, alpha, omega, n0, nres, tol;
  T ta, to, tb;       // alpha, omega, beta in the vector type
  int done, its;
};

// Grid-wide sums of NV <= 2 values per thread, in two parts so that work no other block needs
// can run between a block's arrival and its wait.  begin: four warps per value add a quarter
// of the block's columns each (4 + 5 dependent adds; one warp took 15 + 5), one lane adds the
// quarters, stores the block's partial and arrives.  end: that lane polls, warp 0 adds the
// partials of all blocks in block order (all blocks run the same operations on the same
// partials, so all obtain the same bits) and its first lane runs take(totals, ok).  The partials
// alternate between two buffers (a block can run at most one sum ahead of another).  TURN: one warp
// adds a block's columns, and a lane its partials, one after the other.
template <int NV, bool TURN, class T>
__device__ __forceinline__ unsigned int bicg_sums_begin(BicgShared<T>& sh, const double (&v)[NV], double* part, int buf,
                                                        GridBar* bar) {
  const int G = gridDim.x, nt = blockDim.x;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < NV; ++q) sh.col[q][threadIdx.x] = v[q];
  __syncthreads();
  for (int u = w; u < 4 * NV; u += nt >> 5) {
    if ((u & 3) * 32 >= nt) {   // blocks of fewer than 128 threads: no columns in this quarter
      if (lane == 0) sh.quarter[u >> 2][u & 3] = 0.0;
      continue;
    }
    const double* c = sh.col[u >> 2];
    double t = 0.0;
    if (!TURN)
      for (int j = (u & 3) * 32 + lane; j < nt; j += 128) t += c[j];
    else if ((u & 3) == 0)   // the other quarters are 0
      for (int j = lane; j < nt; j += 32) t += c[j];
    t = warp_sum(t);
    if (lane == 0) sh.quarter[u >> 2][u & 3] = t;
  }
  __syncthreads();
  unsigned int old = 0u;
  if (w == 0) {
    if (lane < NV)
      part[(size_t)(2 * buf + lane) * G + blockIdx.x] = (sh.quarter[lane][0] + sh.quarter[lane][1]) +
                                                         (sh.quarter[lane][2] + sh.quarter[lane][3]);
    __syncwarp();
    if (lane == 0) old = grid_arrive_thread(bar);
  }
  return old;
}

template <int NV, bool TURN, class F>
__device__ __forceinline__ void bicg_sums_end(const double* part, int& buf, GridBar* bar, unsigned int old,
                                              unsigned long long wait_ns, F&& take) {
  const int G = gridDim.x, lane = threadIdx.x & 31;
  if (threadIdx.x < 32) {
    const bool ok = lane != 0 || grid_poll(bar, old, wait_ns);
    __syncwarp();
    double t[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) {
      const double* pb = part + (size_t)(2 * buf + q) * G;
      t[q] = 0.0;
      for (int b0 = lane; b0 - lane < G; b0 += 160) {
        double x[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) x[u] = b0 + 32 * u < G ? __ldcg(pb + b0 + 32 * u) : 0.0;
        t[q] = TURN ? ((((t[q] + x[0]) + x[1]) + x[2]) + x[3]) + x[4] : t[q] + (((x[0] + x[1]) + (x[2] + x[3])) + x[4]);
      }
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) t[q] = warp_sum(t[q]);
    if (lane == 0) take(t, ok);
  }
  buf ^= 1;
  __syncthreads();
}

// The caller's update of a solve's last pass (KrylovEpilogue) at row i.
__device__ __forceinline__ void krylov_update(const KrylovEpilogue& ep, int64_t i, double xi) {
  const double ui = ep.u[i] + ep.omega * xi;
  ep.u[i] = ui;
  if (ep.pair) ep.pair[i] = split_pair(ui);
  if (ep.a) {
    const double uoi = ep.uo[i];
    ep.a[i] = ui - uoi;
    ep.s[i] = ui + uoi;
  }
}
// In the graph form of the fixed point (ep.fp_sc) the solve's launch first decides whether the
// loop goes on (fp_stop.cuh).  True: solve.
__device__ __forceinline__ bool fp_goes_on(const KrylovEpilogue& ep) {
  if (!ep.fp_sc) return true;
  return fp_decide(static_cast<volatile double*>(ep.fp_sc), [&] { return final_sum(ep.part, ep.npart); },
                   [&](bool go) { cudaGraphSetConditional(ep.loop, go ? 1u : 0u); });
}
// The fixed-point loop's count of a correction (one thread of the solve's launch).
__device__ __forceinline__ void krylov_count(const KrylovEpilogue& ep, int its, bool berr, bool broke) {
  double* f = ep.fp_sc;
  if (!f) return;
  f[F_CORR] += 1.0;
  f[F_INNER] += (double)its;
  if (berr || broke) f[F_STATUS] = 2.0;
  if (berr) f[F_TIMEOUT] = 1.0;
}

// SM: the six vectors in shared memory.  TURN: the sums in one order (bicg_fused_launch).
template <int KT, class T, bool SM, bool TURN>
__global__ void __launch_bounds__(kFusedBlock, 1) k_bicg_fused(Offsets of, const T* __restrict__ B,
                                                               const T* __restrict__ dinv, T* ph, T* sg,
                                                               BicgArgs<T> a) {
  const int K = KT > 0 ? KT : of.K;
  const int64_t N = a.N, G = gridDim.x;
  const int64_t i0 = N * blockIdx.x / G;
  const int nrow = (int)(N * (blockIdx.x + 1) / G - i0), nt = blockDim.x, tid = threadIdx.x;
  __shared__ BicgShared<T> sh;
  extern __shared__ __align__(16) char dyn[];
  T* const loc = SM ? reinterpret_cast<T*>(dyn) : a.loc + i0;
  const size_t ls = SM ? (size_t)a.rows : a.vstride;
  T *const r = loc, *const rh = loc + ls, *const p = loc + 2 * ls, *const v = loc + 3 * ls, *const t = loc + 4 * ls,
           *const x = loc + 5 * ls;
  ph += i0;
  sg += i0;
  dinv += i0;
  const double* rhs = a.rhs + i0;
  const T* Bi = B + i0;
  int buf = 0;
  if (!fp_goes_on(a.ep)) return;
  double a1[1], a2[2];
  // y = B g at row q
  auto product = [&](const T* g, int q) {
    T y = 0;
#pragma unroll
    for (int k = 0; k < K; ++k) y = fma(Bi[k * N + q], g[q + of.o[k]], y);
    return y;
  };
  // r = rhs, rhat = r, x = v = 0, rho = (r, r); and the first iteration's p update
  // (beta = 0 and p = v = 0 before it: p = r + 0, phat = D^{-1} p), so that
  // iteration needs no pass and no barrier of its own before its product
  T a0 = 0;
  for (int q = tid; q < nrow; q += nt) {
    const T ri = (T)rhs[q];
    x[q] = 0;
    r[q] = ri;
    rh[q] = ri;
    v[q] = 0;
    const T pi = ri + (T)0;   // as r + 0 * (0 - 1 * 0) rounds: -0 becomes +0
    p[q] = pi;
    ph[q] = dinv[q] * pi;
    a0 = fma(ri, ri, a0);
  }
  a1[0] = to_dbl(a0);
  unsigned int old = bicg_sums_begin<1, TURN>(sh, a1, a.part, buf, a.bar);
  bicg_sums_end<1, TURN>(a.part, buf, a.bar, old, a.wait_ns, [&](const double (&s)[1], bool ok) {
    sh.rho = s[0];
    sh.n0 = sh.nres = sqrt(s[0]);
    sh.tol = fmax(a.atol, a.rtol * sh.n0);
    sh.alpha = sh.omega = 1.0;
    sh.its = 0;
    sh.done = !isfinite(sh.n0) || !ok ? 2 : (sh.n0 < sh.tol ? 1 : (a.maxit <= 0 ? 4 : 0));
  });
  for (bool first = true; sh.done == 0; first = false) {
    // p = r + beta (p - omega v), phat = D^{-1} p (the first iteration's came with r)
    if (!first) {
      const T tb = sh.tb, to = sh.to;
      for (int q = tid; q < nrow; q += nt) {
        const T pi = r[q] + tb * (p[q] - to * v[q]);
        p[q] = pi;
        ph[q] = dinv[q] * pi;
      }
      grid_barrier(a.bar, a.wait_ns);
    }
    // v = B phat, alpha = rho / (rhat, v)
    a0 = 0;
    for (int q = tid; q < nrow; q += nt) {
      const T y = product(ph, q);
      v[q] = y;
      a0 = fma(rh[q], y, a0);
    }
    a1[0] = to_dbl(a0);
    old = bicg_sums_begin<1, TURN>(sh, a1, a.part, buf, a.bar);
    bicg_sums_end<1, TURN>(a.part, buf, a.bar, old, a.wait_ns, [&](const double (&s)[1], bool ok) {
      sh.alpha = sh.rho / s[0];
      sh.ta = (T)sh.alpha;
      if (!isfinite(sh.alpha) || s[0] == 0.0 || !ok) sh.done = 2;
    });
    if (sh.done) break;
    // s = r - alpha v (in place of r), shat = D^{-1} s, ||s||
    const T ta = sh.ta;
    a0 = 0;
    for (int q = tid; q < nrow; q += nt) {
      const T si = r[q] - ta * v[q];
      r[q] = si;
      sg[q] = dinv[q] * si;
      a0 = fma(si, si, a0);
    }
    a1[0] = to_dbl(a0);
    old = bicg_sums_begin<1, TURN>(sh, a1, a.part, buf, a.bar);
    bicg_sums_end<1, TURN>(a.part, buf, a.bar, old, a.wait_ns, [&](const double (&s)[1], bool ok) {
      const double ns = sqrt(s[0]);
      if (!isfinite(ns) || !ok) {
        sh.done = 2;
      } else if (ns < sh.tol) {   // converged at s
        sh.nres = ns;
        sh.its += 1;
        sh.done = 3;
      }
    });
    if (sh.done) break;
    // t = B shat, omega = (t, s) / (t, t)
    T b0 = 0, b1 = 0;
    for (int q = tid; q < nrow; q += nt) {
      const T y = product(sg, q);
      t[q] = y;
      b0 = fma(y, r[q], b0);
      b1 = fma(y, y, b1);
    }
    a2[0] = to_dbl(b0);
    a2[1] = to_dbl(b1);
    old = bicg_sums_begin<2, TURN>(sh, a2, a.part, buf, a.bar);
    bicg_sums_end<2, TURN>(a.part, buf, a.bar, old, a.wait_ns, [&](const double (&s)[2], bool ok) {
      sh.omega = s[0] / s[1];
      sh.to = (T)sh.omega;
      if (!isfinite(sh.omega) || s[1] == 0.0 || !ok) sh.done = 2;
    });
    if (sh.done) break;
    // r = s - omega t, ||r||, (rhat, r); x += alpha phat + omega shat while the sums
    // complete (no other block reads x)
    const T tom = sh.to;
    b0 = 0;
    b1 = 0;
    for (int q = tid; q < nrow; q += nt) {
      const T ri = r[q] - tom * t[q];
      r[q] = ri;
      b0 = fma(ri, ri, b0);
      b1 = fma(rh[q], ri, b1);
    }
    a2[0] = to_dbl(b0);
    a2[1] = to_dbl(b1);
    old = bicg_sums_begin<2, TURN>(sh, a2, a.part, buf, a.bar);
    for (int q = tid; q < nrow; q += nt) x[q] = x[q] + ta * ph[q] + tom * sg[q];
    bicg_sums_end<2, TURN>(a.part, buf, a.bar, old, a.wait_ns, [&](const double (&s)[2], bool ok) {
      const double nr = sqrt(s[0]), rho_old = sh.rho;
      sh.nres = nr;
      sh.rho = s[1];
      sh.tb = (T)((s[1] / rho_old) * (sh.alpha / sh.omega));
      sh.its += 1;
      if (!isfinite(nr) || !ok) sh.done = 2;
      else if (nr < sh.tol) sh.done = 1;
      else if (sh.its >= a.maxit) sh.done = 4;
    });
  }
  const int done = sh.done == 3 ? 1 : sh.done;
  const T last = sh.done == 3 ? sh.ta : (T)0;   // converged at s: x += alpha phat
  const bool upd = a.ep.u != nullptr && done != 2;
  for (int q = tid; q < nrow; q += nt) {
    const T xq = last != (T)0 ? x[q] + last * ph[q] : x[q];
    const double xi = to_dbl(xq);
    a.xout[i0 + q] = xi;
    if (upd) krylov_update(a.ep, i0 + q, xi);
  }
  if (blockIdx.x == 0 && tid == 0) {   // the solver's scalars
    volatile int* berr = &a.bar->err;
    double* sc = a.sc;
    sc[S_TOL] = sh.tol;
    sc[S_N0] = sh.n0;
    sc[S_NRES] = sh.nres;
    sc[S_ITS] = (double)sh.its;
    sc[S_ALPHA] = sh.alpha;
    sc[S_OMEGA] = sh.omega;
    sc[S_RHO] = sh.rho;
    sc[S_DONE] = *berr ? 2.0 : (double)done;
    sc[S_BERR] = *berr ? 1.0 : 0.0;
    krylov_count(a.ep, sh.its, *berr != 0, done == 2);
  }
}

// ---- GMRES(m), right Jacobi preconditioning, classical Gram-Schmidt with one
// re-orthogonalisation pass, as one persistent cooperative launch ----------------
//
// A whole solve (all restart cycles) is one launch.  With a launch per pass the solve
// was bound by launches: five per Arnoldi step (7 to 21 us each on P1 49^3 to 129^3
// for 1 to 10 us of traffic), and a captured cycle ran all m = 20 steps although the
// stationary solves stop after 5 to 10 of them (the rest returned at once, but were
// launched).  Here a step is two or three grid-wide sums, and a solve stops where it stops.
// Measured on one GB300 against the launches per pass, a stationary MC solve (omega = 0.5, inner
// rtol 1e-2) of Q1 27x21x33 in double: 289 -> 59 ms, the same iteration counts.  The second
// projection is taken in nearly all steps (3431 of 3441 there): with the Jacobi preconditioner
// B D^{-1} has a unit diagonal, so that w is mostly v_k.  The single-precision solve has a kernel of
// its own below (k_gm_single).
//
// Layout.  Block b owns a contiguous range of rows (a multiple of 32) for every pass, so
// everything but the product's gather of z is local to a block:
//  * w (the new direction) stays in shared memory between the passes of a step, and so
//    do the basis vectors where all m + 1 of a block fit (up to 928 rows a block at m = 20);
//    otherwise they are in global memory, read 16 bytes per load, four vectors at a
//    time, each once per pass;
//  * the basis vectors are stored unnormalised with their scale 1 / ||v_q|| beside them
//    (in `scale`), so no pass only normalises; z = D^{-1} v_k is the one vector other
//    blocks read, written by the pass that completes v_k.
// Scalars.  A double operation by all warps of an SM costs 16 cycles per warp on the
// FP64 pipe, so the Hessenberg column, Givens rotations and tests run in one warp of
// every block, redundantly and in the same order: every block obtains the same bits and
// takes the same branches without another barrier.  That warp owns no rows: the column
// of step k is rotated while the other warps project and then while they form the next
// product, so the chain of dependent double operations (4 us a step when the block waited
// for it) is hidden; the product that follows a cycle's last step is formed in vain.
//
// Per Arnoldi step k (V holds v_0 .. v_k):
//  (1) w = B z, the dots of V and w, ||w||^2                          -> grid sums
//      DGKS test: if ||w - V h1||^2 = ||w||^2 - ||h1||^2 >= ||w||^2 / 2 little of w lay in
//      the basis and a second projection would change nothing worth keeping;
//      otherwise w -= V h1, h2 = V^T w, ||w||^2                      -> grid sums
//  (2) v_{k+1} = w - V h, z = D^{-1} v_{k+1}, ||v_{k+1}||^2          -> grid sum, or a barrier
//      (gm_second_norm)
//      Hessenberg column, rotations, |g[k+1]|, the end-of-cycle test.
// Threads of a block, at most: with the basis in shared memory (few rows: 96 registers keep
// more of a row's loads in flight), and in global memory (64 registers).
constexpr int kGmBlockS = 544, kGmBlock = 1024;
constexpr int kGmMinCompute = 224;         // threads with rows: few-row blocks still need warps that poll
constexpr int kGmUnit = 32;                // rows of a block come in multiples of this
constexpr int kGmQ = kMaxRestart + 2;      // values of one exchange: k + 1 dots and a norm
// Shared memory for w and V: what is left of 228 KB stays L1, where the product's gather
// of z lives (three bands of a block's rows: ~90 KB suffice up to the sizes that fit).
constexpr size_t kGmSmem = 160 * 1024;

struct GmArgs {
  int64_t N;
  double* sc;
  const double* rhs;
  double* xout;
  size_t vstride;
  GridBar* bar;
  double* part;
  double atol, rtol;
  int maxit, m, compute, rows;
  bool w_in_smem;
  KrylovEpilogue ep;
  unsigned long long wait_ns;
};

// 16 bytes of a vector.
template <class T>
struct alignas(16) Pack {
  static constexpr int W = 16 / sizeof(T);
  T e[W];
};

// Totals over a warp of four values per lane in six adds (a butterfly that halves the values
// with the lanes, then sums) instead of twenty; lane l returns the total of value l >> 3
// (bits 4 and 3 of the lane are bits 1 and 0 of the value).
template <class T>
__device__ __forceinline__ T warp_sum4(const T (&v)[4]) {
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8;
  T a[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const T send = b4 ? v[j] : v[j + 2], keep = b4 ? v[j + 2] : v[j];
    a[j] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
  }
  const T send = b3 ? a[0] : a[1], keep = b3 ? a[1] : a[0];
  T t = keep + __shfl_xor_sync(0xffffffffu, send, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Scalars of a solve, one copy per block.
struct GmScalars {
  double tot[kGmQ];                    // totals of the last exchange
  double nrm2;                         // ||v_{k+1}||^2
  double scale[kMaxRestart + 1];       // 1 / ||v_q||
  double h1[kMaxRestart], h2[kMaxRestart];
  double cs[kMaxRestart], sn[kMaxRestart], g[kMaxRestart + 1], y[kMaxRestart];
  double H[kMaxRestart][kMaxRestart];  // H[row][col], upper triangle after the rotations
  double run;                          // running entry of the column being rotated
  double nres, n0, tol;
  int its, cycles, done, cycle_done, skip, sum_norm;
};
template <class T>
struct GmVectorScalars : GmScalars {
  T hs[kMaxRestart];                   // coefficients of the projection at hand, in the vector type
  T ih;                                // factor of w in the projection
};
template <class T>
struct GmShared : GmVectorScalars<T> {
  T red[kGmBlock / 32][kGmQ + 3];      // the warps' sums (rows padded against bank conflicts)
  // value q of the block
  __device__ __forceinline__ T value(int q, int nw) const {
    T s0 = 0, s1 = 0, s2 = 0, s3 = 0;   // four chains: the adds of one are serial
    int u = 0;
#pragma unroll 1
    for (; u + 3 < nw; u += 4) {
      s0 += red[u][q];
      s1 += red[u + 1][q];
      s2 += red[u + 2][q];
      s3 += red[u + 3][q];
    }
    for (; u < nw; ++u) s0 += red[u][q];
    return (s0 + s1) + (s2 + s3);
  }
};

// The total over a warp of one partial of G per slot, p[0 .. G), in a fixed order.
__device__ __forceinline__ double gm_total(const double* p, int G) {
  const int lane = threadIdx.x & 31;
  double x[5];   // G <= 160
#pragma unroll
  for (int u = 0; u < 5; ++u) x[u] = lane + 32 * u < G ? __ldcg(p + lane + 32 * u) : 0.0;
  const double t = ((x[0] + x[1]) + (x[2] + x[3])) + x[4];
  return warp_sum(t);
}

// A grid-wide sum of nq values and a barrier: warp 0 stores the block's values, value(q), its
// first lane arrives and polls; then warp q adds all blocks' partials of value q into sh.tot
// (the same bits in every block), and `take()` runs in warp 0 (with nq <= 1 before the block meets
// again, in the same warp).  Memory: the
// block's threads meet, so that lane's fence releases what they wrote; it polls with acquire
// loads, and the block meets again before anyone uses what `take` stored or what other
// blocks wrote.  The partials alternate between two buffers (a block can run at most one
// sum ahead of another).
template <class V, class F>
__device__ __forceinline__ void gm_exchange(GmScalars& sh, int nq, const GmArgs& a, int& buf, V&& value, F&& take) {
  const int G = gridDim.x, lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  double* pb = a.part + (size_t)buf * kGmQ * G;
  buf ^= 1;
  __syncthreads();   // what value() reads is complete
  if (wp == 0) {
#pragma unroll 1
    for (int q = lane; q < nq; q += 32) pb[(size_t)q * G + blockIdx.x] = value(q);
    __syncwarp();
    if (lane == 0) grid_poll(a.bar, grid_arrive_thread(a.bar), a.wait_ns);
    __syncwarp();
  }
  if (nq > 1) __syncthreads();
  if (nq > 1 || wp == 0) {
#pragma unroll 1
    for (int q = wp; q < nq; q += blockDim.x >> 5) {
      const double t = gm_total(pb + (size_t)q * G, G);
      if (lane == 0) sh.tot[q] = t;
    }
  }
  if (nq > 1) __syncthreads();
  if (wp == 0) {
    __syncwarp();
    take();
  }
  __syncthreads();
}
__device__ __forceinline__ void gm_barrier(GmScalars& sh, const GmArgs& a, int& buf) {
  gm_exchange(sh, 0, a, buf, [](int) { return 0.0; }, [] {});
}

// The warps' sums of one value per thread, as value q of sh.red.
template <class T>
__device__ __forceinline__ void gm_put(GmShared<T>& sh, T v, int q) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0) sh.red[threadIdx.x >> 5][q] = v;
}

// Run f(NQ as a constant, q) over q = 0 .. n - 1 in steps of four and a rest of one to three:
// loops over the basis without a predicate per vector (which cost the registers that hold
// the loads in flight).
template <class F>
__device__ __forceinline__ void by_fours(int n, F&& f) {
  int q = 0;
#pragma unroll 1
  for (; q + 4 <= n; q += 4) f(std::integral_constant<int, 4>{}, q);
  if (n - q == 3) f(std::integral_constant<int, 3>{}, q);
  else if (n - q == 2) f(std::integral_constant<int, 2>{}, q);
  else if (n - q == 1) f(std::integral_constant<int, 1>{}, q);
}

// The warps' dots (w, v_q), q <= k, as values 0 .. k of sh.red, and (w, w) as value k + 1.
// ng: groups of 16 bytes in a block's rows; nw: warps that hold any.
template <class T>
__device__ __forceinline__ void gm_dots(GmShared<T>& sh, const T* w, const T* V, size_t vs, int ng, int nw, int nt,
                                        int k) {
  constexpr int W = Pack<T>::W;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  if (wp >= nw) return;
  by_fours(k + 1, [&](auto nq, int q0) {
    constexpr int NQ = decltype(nq)::value;
    T acc[4] = {0, 0, 0, 0};
    const T* Vq = V + (size_t)q0 * vs;
#pragma unroll 1
    for (int g = threadIdx.x; g < ng; g += nt) {
      const Pack<T> wi = *reinterpret_cast<const Pack<T>*>(w + g * W);
      Pack<T> v[NQ];
#pragma unroll
      for (int j = 0; j < NQ; ++j) v[j] = *reinterpret_cast<const Pack<T>*>(Vq + j * vs + g * W);
#pragma unroll
      for (int j = 0; j < NQ; ++j)
#pragma unroll
        for (int e = 0; e < W; ++e) acc[j] = fma(wi.e[e], v[j].e[e], acc[j]);
    }
    const T t = warp_sum4(acc);
    if ((lane & 7) == 0 && (lane >> 3) < NQ) sh.red[wp][q0 + (lane >> 3)] = t;
  });
  T nrm = 0;
#pragma unroll 1
  for (int g = threadIdx.x; g < ng; g += nt) {
    const Pack<T> wi = *reinterpret_cast<const Pack<T>*>(w + g * W);
#pragma unroll
    for (int e = 0; e < W; ++e) nrm = fma(wi.e[e], wi.e[e], nrm);
  }
  gm_put(sh, nrm, k + 1);
}

// ih w - sum_q hs[q] v_q (q <= k) of group g.
template <class T>
__device__ __forceinline__ Pack<T> gm_project(const GmVectorScalars<T>& sh, T ih, const T* w, const T* V, size_t vs, int g,
                                              int k) {
  constexpr int W = Pack<T>::W;
  Pack<T> wi = *reinterpret_cast<const Pack<T>*>(w + g * W);
#pragma unroll
  for (int e = 0; e < W; ++e) wi.e[e] *= ih;
  by_fours(k + 1, [&](auto nq, int q0) {
    constexpr int NQ = decltype(nq)::value;
    Pack<T> v[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) v[j] = *reinterpret_cast<const Pack<T>*>(V + (size_t)(q0 + j) * vs + g * W);
#pragma unroll
    for (int j = 0; j < NQ; ++j)
#pragma unroll
      for (int e = 0; e < W; ++e) wi.e[e] -= sh.hs[q0 + j] * v[j].e[e];
  });
  return wi;
}

// The passes over a block's rows.
// w = ih w - V h.
template <class T>
__device__ __forceinline__ void gm_reproject(const GmShared<T>& sh, T* w, const T* V, size_t vs, int ng, int nt, int k) {
  const T ih = sh.ih;
#pragma unroll 1
  for (int g = threadIdx.x; g < ng; g += nt)
    *reinterpret_cast<Pack<T>*>(w + g * Pack<T>::W) = gm_project(sh, ih, w, V, vs, g, k);
}
// v_{k+1} = ih w - V h, z = D^{-1} v_{k+1} at the block's rows, and the warps' sums of
// ||v_{k+1}||^2.
template <class T>
__device__ __forceinline__ void gm_complete(GmShared<T>& sh, const T* w, T* V, size_t vs, int ng, int nt, int k,
                                         const T* __restrict__ dinv, T* z, int nrow) {
  constexpr int W = Pack<T>::W;
  const T ih = sh.ih;
  T* vn = V + (size_t)(k + 1) * vs;
  T nrm = 0;
#pragma unroll 1
  for (int g = threadIdx.x; g < ng; g += nt) {
    const Pack<T> v = gm_project(sh, ih, w, V, vs, g, k);
    *reinterpret_cast<Pack<T>*>(vn + g * W) = v;
#pragma unroll
    for (int e = 0; e < W; ++e) {
      const int r = g * W + e;
      if (r < nrow) z[r] = dinv[r] * v.e[e];
      nrm = fma(v.e[e], v.e[e], nrm);
    }
  }
  gm_put(sh, nrm, 0);
}
// x (+)= D^{-1} sum_q hs[q] v_q, q < ku (sh.ih = 0 and hs negated: the projection's form).
template <class T>
__device__ __forceinline__ void gm_update(const GmShared<T>& sh, const T* w, const T* V, size_t vs, int ng, int nt, int ku,
                                       const T* __restrict__ dinv, T* x, int nrow, bool have_x) {
  constexpr int W = Pack<T>::W;
#pragma unroll 1
  for (int g = threadIdx.x; g < ng; g += nt) {
    const Pack<T> s = gm_project(sh, (T)0, w, V, vs, g, ku - 1);
#pragma unroll
    for (int e = 0; e < W; ++e) {
      const int r = g * W + e;
      if (r < nrow) {
        const T d = dinv[r] * s.e[e];
        x[r] = have_x ? x[r] + d : d;
      }
    }
  }
}

// Column k of the Hessenberg matrix, in the scalar warp: the earlier rotations (while the
// other warps complete v_{k+1}).  The running entry c <- -sn_q c + cs_q b_q is one dependent
// multiply-add per rotation; lane q forms the products and its entry of the column.
__device__ __forceinline__ void gm_rotate(GmScalars& sh, int k) {
  const int q = threadIdx.x & 31;
  double cb = 0.0, sb = 0.0, cs = 0.0, sn = 0.0, mine = 0.0;
  if (q < k) {
    const double b = sh.h1[q + 1] + sh.h2[q + 1];
    cs = sh.cs[q];
    sn = sh.sn[q];
    cb = cs * b;
    sb = sn * b;
  }
  double c = sh.h1[0] + sh.h2[0];
#pragma unroll 1
  for (int r = 0; r < k; ++r) {
    if (q == r) mine = c;
    c = fma(-__shfl_sync(0xffffffffu, sn, r), c, __shfl_sync(0xffffffffu, cb, r));
  }
  if (q < k) sh.H[q][k] = fma(cs, mine, sb);
  if (q == 0) sh.run = c;
}
// ||v_{k+1}||^2 after a second projection, in the same warp: w was almost orthogonal to the basis, so
// that ||w - V h2||^2 = ||w||^2 - ||h2||^2 needs no sum of its own (3 us of a step of 18).  Only where
// less than 2^-10 of ||w||^2 is taken away: the difference is then as exact as the sum ||w||^2.
__device__ __forceinline__ void gm_second_norm(GmScalars& sh, int k) {
  const int q = threadIdx.x & 31;
  const double h = !sh.skip && q <= k ? sh.h2[q] : 0.0, p = warp_sum(h * h);
  if (q != 0) return;
  sh.sum_norm = sh.skip || !(p <= 0x1p-10 * sh.nrm2);
  if (!sh.sum_norm) sh.nrm2 -= p;
}
// ... then, from ||v_{k+1}||^2, the new rotation, the residual estimate and the
// end-of-cycle test (while they form the next product).
__device__ __forceinline__ void gm_column(GmScalars& sh, int k, const GmArgs& a, bool berr) {
  const double n2 = sh.nrm2, c = sh.run, den2 = fma(c, c, n2);
  const double inv = rsqrt(n2), hk1 = n2 > 0.0 ? n2 * inv : sqrt(n2);
  const double rden = rsqrt(den2), den = den2 > 0.0 ? den2 * rden : sqrt(den2);
  const double sk = hk1 * rden, ck = c * rden;
  sh.cs[k] = ck;
  sh.sn[k] = sk;
  sh.H[k][k] = den;
  const double gk = sh.g[k], gn = -sk * gk;
  sh.g[k + 1] = gn;
  sh.g[k] = ck * gk;
  sh.its += 1;
  sh.nres = fabs(gn);
  sh.scale[k + 1] = inv;
  if (!isfinite(den) || den == 0.0 || berr) sh.done = 2;
  else if (fabs(gn) < sh.tol || sh.its >= a.maxit || k + 1 == a.m || hk1 == 0.0) sh.cycle_done = 1;
}

// H y = g for the leading ku columns (from the last; lane c keeps g[c]), in one warp.
__device__ __forceinline__ void gm_triangle(GmScalars& sh, int ku) {
  const int c = threadIdx.x & 31;
  double gc = c < ku ? sh.g[c] : 0.0;
  const double inv = c < ku ? 1.0 / sh.H[c][c] : 0.0;
#pragma unroll 1
  for (int q = ku - 1; q >= 0; --q) {
    const double yq = __shfl_sync(0xffffffffu, gc * inv, q);
    if (c == q) sh.y[q] = yq;
    if (c < q) gc = fma(-sh.H[c][q], yq, gc);
  }
  __syncwarp();
}

// w = B z over a block's rows (B, z, w at the block's first row).  The row's addresses are
// formed inside the loop, from a stride and a base the compiler cannot see through: hoisted
// out of it they took 4 K registers, and the row's 2 K loads went out a few at a time.
// STREAM: the matrix goes past L2 (evict first), which the basis vectors then keep (measured at
// P1 129^3 in single precision with the rows of a block in one range: product 26.8 -> 24.9 us, dots
// 13.9 -> 10.4 us).
template <int KT, bool STREAM, class T>
__device__ __forceinline__ void gm_product(const Offsets& of, int64_t N, const T* __restrict__ B, const T* z, T* w,
                                           int nrow, int nt) {
  const int K = KT > 0 ? KT : of.K;
#pragma unroll 1
  for (int r = threadIdx.x; r < nrow; r += nt) {
    int64_t n = N;
    const T* zr = z + r;
    asm volatile("" : "+l"(n), "+l"(zr));
    const T* br = B + r;
    T s = 0;
#pragma unroll
    for (int q = 0; q < K; ++q) s = fma(STREAM ? __ldcs(br + q * n) : br[q * n], zr[of.o[q]], s);
    w[r] = s;
  }
}

// The solver's scalars at the end of a solve.
__device__ __forceinline__ void gm_report(const GmScalars& sh, const GmArgs& a, bool berr) {
  double* sc = a.sc;
  sc[S_N0] = sh.n0;
  sc[S_TOL] = sh.tol;
  sc[S_NRES] = sh.nres;
  sc[S_BETA] = sh.nres;
  sc[S_ITS] = (double)sh.its;
  sc[S_CYCLES] = (double)sh.cycles;
  sc[S_DONE] = berr ? 2.0 : (double)sh.done;
  sc[S_BERR] = berr ? 1.0 : 0.0;
  krylov_count(a.ep, sh.its, berr, sh.done == 2);
}

// VS: the basis in shared memory.
template <int KT, class T, bool VS>
__global__ void __launch_bounds__(VS ? kGmBlockS : kGmBlock, 1) k_gm_fused(Offsets of, const T* __restrict__ B,
                                                             const T* __restrict__ dinv, T* x, T* z, T* wg, T* Vg,
                                                             GmArgs a) {
  constexpr int W = Pack<T>::W;
  const int64_t N = a.N;
  const int64_t units = (N + kGmUnit - 1) / kGmUnit;
  const int64_t i0 = units * blockIdx.x / gridDim.x * kGmUnit;
  const int64_t i1 = units * (blockIdx.x + 1) / gridDim.x * kGmUnit;
  const int nrow = (int)((i1 < N ? i1 : N) - i0);
  const int nt = a.compute;                       // threads with rows; the last warp has the scalars
  const bool rows_warp = (int)threadIdx.x < nt, scalar = (int)threadIdx.x == nt;   // scalar: its first lane
  const int ng = (nrow + W - 1) / W;              // 16-byte groups; the last one may reach past N
  const int nw = min(nt, (ng + 31) / 32 * 32) / 32;   // warps that hold any
  __shared__ GmShared<T> sh;
  extern __shared__ __align__(16) char dyn[];
  // w (and V) of this block: in shared memory, or at its rows in global memory.  The tail of
  // the last group is zero and stays so (w, V and B z are 0 there).
  T* const w = VS || a.w_in_smem ? reinterpret_cast<T*>(dyn) : wg + i0;
  T* const V = VS ? reinterpret_cast<T*>(dyn) + a.rows : Vg + i0;
  const size_t vs = VS ? (size_t)a.rows : a.vstride;
  for (int r = nrow + threadIdx.x; r < ng * W; r += blockDim.x) w[r] = (T)0;
  volatile int* berr = &a.bar->err;
  int buf = 0;
  auto value = [&](int q) { return sh.value(q, nw); };
  if (!fp_goes_on(a.ep)) return;
  if (scalar) {
    sh.its = 0;
    sh.cycles = 0;
    sh.done = 0;
  }
  bool have_x = false;   // x = 0 until the first cycle's update
  for (;;) {
    // true residual v_0 = rhs - B x, z = D^{-1} v_0, ||v_0||
    if (have_x && rows_warp) gm_product<KT, !VS>(of, N, B + i0, x + i0, w, nrow, nt);
    __syncthreads();
    if (rows_warp) {
      T nrm = 0;
#pragma unroll 1
      for (int g = threadIdx.x; g < ng; g += nt) {
        Pack<T> v;
#pragma unroll
        for (int e = 0; e < W; ++e) {
          const int r = g * W + e;
          v.e[e] = (T)0;
          if (r < nrow) {
            v.e[e] = have_x ? (T)a.rhs[i0 + r] - w[r] : (T)a.rhs[i0 + r];
            z[i0 + r] = dinv[i0 + r] * v.e[e];
          }
          nrm = fma(v.e[e], v.e[e], nrm);
        }
        *reinterpret_cast<Pack<T>*>(V + g * W) = v;
      }
      gm_put(sh, nrm, 0);
    }
    gm_exchange(sh, 1, a, buf, value, [&]() {
      if (threadIdx.x != 0) return;
      const double beta = sqrt(sh.tot[0]);
      if (!have_x) {
        sh.n0 = beta;
        sh.tol = fmax(a.atol, a.rtol * beta);
      }
      sh.cycles += 1;
      sh.nres = beta;
      sh.cycle_done = 0;
      if (!isfinite(beta) || *berr) sh.done = 2;
      else if (beta < sh.tol) sh.done = 1;
      else if (sh.its >= a.maxit) sh.done = 4;
      sh.g[0] = beta;
      sh.scale[0] = 1.0 / beta;
    });
    if (sh.done != 0) break;
    int ku = 0;   // columns of this cycle
    for (int k = 0;; ++k) {
      // (1) w = B z and its dots; meanwhile the scalar warp ends column k - 1
      if (rows_warp) {
        gm_product<KT, !VS>(of, N, B + i0, z + i0, w, nrow, nt);
      } else if (scalar && k > 0) {
        gm_column(sh, k - 1, a, *berr != 0);
      }
      __syncthreads();
      ku = k;
      if (sh.done != 0 || (k > 0 && sh.cycle_done != 0)) break;
      gm_dots(sh, w, V, vs, ng, nw, nt, k);
      // h1 and the projection's coefficients: w stands for w / ||v_k||, v_q for v_q / ||v_q||
      gm_exchange(sh, k + 2, a, buf, value, [&]() {
        const int q = threadIdx.x;
        const double sk = sh.scale[k], ww = sh.tot[k + 1] * (sk * sk);
        double h = 0.0;
        if (q <= k) {
          const double sq = sh.scale[q];
          h = sh.tot[q] * (sq * sk);
          sh.h1[q] = h;
          sh.h2[q] = 0.0;
          sh.hs[q] = (T)(h * sq);
        }
        const double rest = ww - warp_sum(h * h);
        if (q == 0) {
          sh.ih = (T)sk;
          sh.skip = rest >= 0.5 * ww && ww > 0.0;
        }
      });
      if (!sh.skip) {   // second projection: w = w - V h1, h2 = V^T w, ||w||^2
        if (rows_warp) gm_reproject(sh, w, V, vs, ng, nt, k);
        // a thread's dots read the groups it wrote
        gm_dots(sh, w, V, vs, ng, nw, nt, k);
        gm_exchange(sh, k + 2, a, buf, value, [&]() {
          const int q = threadIdx.x;
          if (q <= k) {
            const double sq = sh.scale[q], h = sh.tot[q] * sq;
            sh.h2[q] = h;
            sh.hs[q] = (T)(h * sq);
          }
          if (q == 0) {
            sh.nrm2 = sh.tot[k + 1];
            sh.ih = (T)1;
          }
        });
      }
      // (2) v_{k+1} = w - V h, z = D^{-1} v_{k+1}, ||v_{k+1}||^2; meanwhile the scalar warp
      // rotates column k
      if (rows_warp) {
        gm_complete(sh, w, V, vs, ng, nt, k, dinv + i0, z + i0, nrow);
      } else {
        gm_rotate(sh, k);
        gm_second_norm(sh, k);
      }
      __syncthreads();
      const bool sum = sh.sum_norm;
      gm_exchange(sh, sum ? 1 : 0, a, buf, value, [&]() {
        if (sum && threadIdx.x == 0) sh.nrm2 = sh.tot[0];
      });
    }
    if (sh.done != 0) break;
    // x += D^{-1} sum_q y_q v_q / ||v_q||
    if (threadIdx.x < 32) {
      gm_triangle(sh, ku);
      const int c = threadIdx.x;
      if (c < ku) sh.hs[c] = (T)(-sh.y[c] * sh.scale[c]);
    }
    __syncthreads();
    if (rows_warp) {
      gm_update(sh, w, V, vs, ng, nt, ku, dinv + i0, x + i0, nrow, have_x);
    }
    have_x = true;
    gm_barrier(sh, a, buf);   // the next residual gathers x
  }
  // the solution, and the caller's update unless the solve broke down
  const bool upd = a.ep.u != nullptr && sh.done != 2;
#pragma unroll 1
  for (int r = threadIdx.x; r < nrow; r += blockDim.x) {
    const int64_t i = i0 + r;
    const double xi = have_x ? (double)x[i] : 0.0;
    a.xout[i] = xi;
    if (upd) krylov_update(a.ep, i, xi);
  }
  if (blockIdx.x == 0 && scalar) gm_report(sh, a, *berr != 0);
}

// ---- GMRES(m) on single-precision vectors -----------------------------------------
//
// The same method and launch, but with every single-precision rounding in a fixed place.  The
// damped iteration around a mixed solve amplifies the rounding of its inner solver at isolated
// nodes: with the dots added in another order and the basis unnormalised, whole stationary solves
// moved by 2e-12 to 2e-8 (P1 49^3 and 129^3, the same number of corrections and the same residual).
// So here
//  * the basis vectors are normalised and rounded once, v_k = w (1 / ||w||), z = D^{-1} v_k;
//  * a dot is formed by single-precision strands: rows come in chunks of 256, chunk c adds to strand
//    set c mod (gm_strand_sets * SMs), each of whose 256 strands takes its rows in ascending order by
//    multiply-adds; 32 strands are added by a butterfly, the eight results of a set in turn, and the
//    sets' sums in double.  The order of the double-precision additions is free: their rounding is
//    far below the last bit of the single-precision coefficients they give;
//  * the squares of a new vector's entries are added in single precision along a strand and in
//    double across strands, those of the true residual in double from the first addition.
// gm_strand_sets (per SM) is part of that definition: a result depends on it, and on the device's
// SM count, but not on scheduling or on where the vectors are kept.
// The norm needs a grid-wide sum of its own and z a barrier after it: a step is three sums and a
// barrier where the kernel above takes two and a barrier.  Measured on one GB300 (a kernel per pass ->
// unnormalised in this kernel's place -> this kernel): stationary P1 49^3 511 -> 101 -> 152 ms, 129^3
// 1.75 -> 0.82 -> 1.01 s, a burst of 8 served requests 911 -> 74 -> 98 ms.
//
// Block b owns chunks b, b + G, b + 2 G, ... (G blocks; G = SMs, or fewer when each has at most two
// chunks): the chunks of a strand set are then all in one block, for every number of sets, so that
// w and the basis stay local to it.  In a block of chunks s = 0 .. S - 1 the sets are s mod R, and
// a row's local index is 256 s + its place in the chunk.
constexpr int kGsChunk = 256;
// strand sets per SM of a step with n basis vectors (n <= kMaxRestart)
__host__ __device__ __forceinline__ constexpr int gm_strand_sets(int n) {
  return n <= 4 ? 6 : n <= 12 ? 5 : n <= 16 ? 4 : n <= 20 ? 3 : 2;
}
// values times sets of one exchange, at most
constexpr int gs_most_sums() {
  int most = 0;
  for (int k = 0; k < kMaxRestart; ++k) most = (k + 2) * gm_strand_sets(k + 1) > most ? (k + 2) * gm_strand_sets(k + 1) : most;
  return most;
}
constexpr int kGsSums = gs_most_sums();
constexpr int kGsWarpRows = 128;           // rows of a chunk that a warp takes at once, 16 bytes a lane
constexpr int kGsParts = kGsChunk / 32;    // butterflies of a strand set

struct GsShared : GmVectorScalars<float> {
  float red[kGsSums][kGsParts + 1];      // [q R + r]: the butterflies of value q, set r
  double fold[kGsSums];                  // ... added in turn
  double col[kGmBlock], quarter[4];              // one double per thread, and their sums
};

// A block's rows.
struct GsRows {
  int b, G, nrow;   // nrow: local rows in use
  int64_t N;
  // place in a vector of all rows
  __device__ __forceinline__ int64_t at(int l) const { return l + ((int64_t)b + (int64_t)(G - 1) * (l / kGsChunk)) * kGsChunk; }
};
// Where the local rows of w and of the basis are kept: in shared memory (at their local index), or in
// global memory (at their place among all rows).
__device__ __forceinline__ int64_t gs_at(const GsRows& rw, bool smem, int l) { return smem ? l : rw.at(l); }

// w = B z over the block's rows (see gm_product).
template <int KT, bool STREAM>
__device__ __forceinline__ void gs_product(const Offsets& of, const GsRows& rw, const float* __restrict__ B, const float* z,
                                           float* w, bool ws, int nt) {
  const int K = KT > 0 ? KT : of.K;
#pragma unroll 1
  for (int l = threadIdx.x; l < rw.nrow; l += nt) {
    const int64_t i = rw.at(l);
    int64_t n = rw.N;
    const float* zr = z + i;
    asm volatile("" : "+l"(n), "+l"(zr));
    const float* br = B + i;
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < K; ++q) s = fma(STREAM ? __ldcs(br + q * n) : br[q * n], zr[of.o[q]], s);
    w[ws ? l : i] = s;
  }
}

// The strands of NQ vectors v_0, v_vs, ... with w for 128 rows of strand set r (half h of its
// chunks), four adjacent strands per lane; then the butterflies of 32 strands each: partners at
// distance 16, 8 and 4 are lanes at distance 4, 2 and 1, those at distance 2 and 1 are entries of a
// lane (halving the entries with the lanes, six shuffles instead of twenty).  Every sum has the
// operands of a butterfly over 32 lanes.
template <int NQ>
__device__ __forceinline__ void gs_strands(GsShared& sh, const float* w, int64_t wstep, const float* V, int64_t vstep,
                                           size_t vs, int r, int h, int R, int S, int nrow, int q0) {
  const int lane = threadIdx.x & 31;
  float acc[NQ][4] = {};
  auto add = [&](const float* wp, const float* vp) {
    const Pack<float> wi = *reinterpret_cast<const Pack<float>*>(wp);
    Pack<float> v[NQ];
#pragma unroll
    for (int j = 0; j < NQ; ++j) v[j] = *reinterpret_cast<const Pack<float>*>(vp + j * vs);
#pragma unroll
    for (int j = 0; j < NQ; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[j][e] = fma(wi.e[e], v[j].e[e], acc[j][e]);
  };
  int s = r;
#pragma unroll 1
  for (; s < S - 1; s += R, w += wstep, V += vstep) add(w, V);
  if (s == S - 1 && s * kGsChunk + h * kGsWarpRows + 4 * lane < nrow) add(w, V);   // the last chunk may end early
  const bool b2 = lane & 4, b1 = lane & 2;
#pragma unroll
  for (int j = 0; j < NQ; ++j) {
    float a[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {   // distance 16: entries e (lanes without bit 2) or e + 2
      const float send = b2 ? acc[j][e] : acc[j][e + 2], keep = b2 ? acc[j][e + 2] : acc[j][e];
      a[e] = keep + __shfl_xor_sync(0xffffffffu, send, 4);
    }
    const float send = b1 ? a[0] : a[1], keep = b1 ? a[1] : a[0];
    float t = keep + __shfl_xor_sync(0xffffffffu, send, 2);   // 8: entry (b2, b1)
    t += __shfl_xor_sync(0xffffffffu, t, 1);                  // 4
    t += __shfl_xor_sync(0xffffffffu, t, 4);                  // 2: entries 0 and 2, 1 and 3
    t += __shfl_xor_sync(0xffffffffu, t, 2);                  // 1
    if ((lane & 7) == 0) sh.red[(q0 + j) * R + r][4 * h + (lane >> 3)] = t;
  }
}

// The strand sums of (w, v_q), q <= k, as values 0 .. k, and with `norm` of (w, w) as value k + 1.
// Items: 128 rows of a strand set (both halves of R sets) times a few of the vectors, as many as
// leave an item for every warp.  Every warp with rows calls it.
__device__ __forceinline__ void gs_dots(GsShared& sh, const GsRows& rw, const float* w, bool ws, const float* V, bool vsm,
                                        size_t vs, int R, int S, int nwarp, int k, bool norm) {
  const int units = 2 * R, most = max(1, nwarp / units);
  const int per = min(4, (k + most) / most);                  // ceil((k + 1) / most)
  const int groups = (k + per) / per;                         // ceil((k + 1) / per)
  const int items = units * (groups + (norm ? 1 : 0));
  const int64_t step = (int64_t)R * kGsChunk;
  const int64_t vstep = vsm ? step : step * rw.G, wstep = ws ? step : step * rw.G;
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int it = threadIdx.x >> 5; it < items; it += nwarp) {
    const int u = it % units, gq = it / units, r = u >> 1, h = u & 1;
    const int l = r * kGsChunk + h * kGsWarpRows + 4 * lane;
    const float* wl = w + gs_at(rw, ws, l);
    if (gq == groups) {
      gs_strands<1>(sh, wl, wstep, wl, wstep, 0, r, h, R, S, rw.nrow, k + 1);
      continue;
    }
    const int q0 = gq * per;
    const float* vl = V + (size_t)q0 * vs + gs_at(rw, vsm, l);
    switch (min(per, k + 1 - q0)) {
      case 4: gs_strands<4>(sh, wl, wstep, vl, vstep, vs, r, h, R, S, rw.nrow, q0); break;
      case 3: gs_strands<3>(sh, wl, wstep, vl, vstep, vs, r, h, R, S, rw.nrow, q0); break;
      case 2: gs_strands<2>(sh, wl, wstep, vl, vstep, vs, r, h, R, S, rw.nrow, q0); break;
      default: gs_strands<1>(sh, wl, wstep, vl, vstep, vs, r, h, R, S, rw.nrow, q0);
    }
  }
}
// ... a set's butterflies added in turn (the block).
__device__ __forceinline__ void gs_fold(GsShared& sh, int n) {
  __syncthreads();
  for (int x = threadIdx.x; x < n; x += blockDim.x) {
    float s = 0.f;
#pragma unroll
    for (int u = 0; u < kGsParts; ++u) s += sh.red[x][u];
    sh.fold[x] = widen_exact(s);
  }
}

// The sum of one double per thread with rows, in four warps, as sh.quarter (the block).
__device__ __forceinline__ void gs_column(GsShared& sh, int nt) {
  const int wp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (wp >= 4) return;
  double t = 0.0;
  for (int j = wp * 32 + lane; j < nt; j += 128) t += sh.col[j];
  t = warp_sum(t);
  if (lane == 0) sh.quarter[wp] = t;
}
// This thread's part of ||w||^2, a single-precision sum per strand: a warp takes 32 strands.
__device__ __forceinline__ double gs_norm(const GsRows& rw, const float* w, bool ws, int R, int S, int nwarp) {
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)R * kGsChunk * (ws ? 1 : rw.G);
  double sum = 0.0;
#pragma unroll 1
  for (int u = threadIdx.x >> 5; u < R * kGsParts; u += nwarp) {
    const int r = u / kGsParts, l = r * kGsChunk + 32 * (u % kGsParts) + lane;
    const float* p = w + gs_at(rw, ws, l);
    float nrm = 0.f;
    int s = r;
#pragma unroll 4
    for (; s < S - 1; s += R, p += step) nrm = fma(*p, *p, nrm);
    if (s == S - 1 && l + (s - r) * kGsChunk < rw.nrow) nrm = fma(*p, *p, nrm);
    sum += widen_exact(nrm);
  }
  return sum;
}

// VS: the basis in shared memory (then w too).
template <int KT, bool VS>
__global__ void __launch_bounds__(VS ? kGmBlockS : kGmBlock, 1) k_gm_single(Offsets of, const float* __restrict__ B,
                                                                const float* __restrict__ dinv, float* x, float* z,
                                                                float* wg, float* Vg, GmArgs a) {
  constexpr int W = Pack<float>::W;
  const int64_t chunks = (a.N + kGsChunk - 1) / kGsChunk;
  GsRows rw;
  rw.b = blockIdx.x;
  rw.G = gridDim.x;
  rw.N = a.N;
  const int S = (int)((chunks - rw.b + rw.G - 1) / rw.G);
  rw.nrow = S * kGsChunk;
  if ((chunks - 1) % rw.G == rw.b) rw.nrow -= (int)(chunks * kGsChunk - a.N);   // it owns the last chunk
  const int nt = a.compute, nwarp = nt >> 5;      // threads with rows; the last warp has the scalars
  const bool rows_warp = (int)threadIdx.x < nt, scalar = (int)threadIdx.x == nt;   // scalar: its first lane
  const int ng = (rw.nrow + W - 1) / W;           // 16-byte groups; the last one may reach past N
  __shared__ GsShared sh;
  extern __shared__ __align__(16) char dyn[];
  const bool ws = VS || a.w_in_smem;
  float* const w = ws ? reinterpret_cast<float*>(dyn) : wg;
  float* const V = VS ? reinterpret_cast<float*>(dyn) + a.rows : Vg;
  const size_t vs = VS ? (size_t)a.rows : a.vstride;
  for (int l = rw.nrow + threadIdx.x; l < ng * W; l += blockDim.x) w[gs_at(rw, ws, l)] = 0.f;   // and stays so
  volatile int* berr = &a.bar->err;
  int buf = 0;
  if (!fp_goes_on(a.ep)) return;
  if (scalar) {
    sh.its = 0;
    sh.cycles = 0;
    sh.done = 0;
  }
  // w -= sum_q hs[q] v_q, q <= k
  auto project = [&](int k) {
#pragma unroll 1
    for (int g = threadIdx.x; g < ng; g += nt) {
      float* wl = w + gs_at(rw, ws, g * W);
      *reinterpret_cast<Pack<float>*>(wl) = gm_project(sh, 1.f, wl, V + gs_at(rw, VS, g * W), vs, 0, k);
    }
  };
  // v_q = ih w, z = D^{-1} v_q
  auto normalise = [&](int q) {
    const float ih = sh.ih;
    float* vq = V + (size_t)q * vs;
#pragma unroll 1
    for (int g = threadIdx.x; g < ng; g += nt) {
      const int l = g * W;
      const int64_t i = rw.at(l);
      Pack<float> v = *reinterpret_cast<const Pack<float>*>(w + (ws ? l : i));
#pragma unroll
      for (int e = 0; e < W; ++e) {
        v.e[e] *= ih;
        if (l + e < rw.nrow) z[i + e] = dinv[i + e] * v.e[e];
      }
      *reinterpret_cast<Pack<float>*>(vq + (VS ? l : i)) = v;
    }
  };
  auto norm_value = [&](int) { return (sh.quarter[0] + sh.quarter[1]) + (sh.quarter[2] + sh.quarter[3]); };
  bool have_x = false;   // x = 0 until the first cycle's update
  for (;;) {
    // true residual w = rhs - B x and its norm, v_0 = w / ||w||
    if (have_x && rows_warp) gs_product<KT, !VS>(of, rw, B, x, w, ws, nt);
    if (rows_warp) {   // a thread's own rows
      double nrm = 0.0;
#pragma unroll 1
      for (int l = threadIdx.x; l < rw.nrow; l += nt) {
        const int64_t i = rw.at(l);
        float* wl = w + (ws ? l : i);
        const float v = have_x ? (float)a.rhs[i] - *wl : (float)a.rhs[i];
        *wl = v;
        nrm += widen_exact(v * v);
      }
      sh.col[threadIdx.x] = nrm;
    }
    gs_column(sh, nt);
    gm_exchange(sh, 1, a, buf, norm_value, [&]() {
      if (threadIdx.x != 0) return;
      const double beta = sqrt(sh.tot[0]);
      if (!have_x) {
        sh.n0 = beta;
        sh.tol = fmax(a.atol, a.rtol * beta);
      }
      sh.cycles += 1;
      sh.nres = beta;
      sh.cycle_done = 0;
      if (!isfinite(beta) || *berr) sh.done = 2;
      else if (beta < sh.tol) sh.done = 1;
      else if (sh.its >= a.maxit) sh.done = 4;
      sh.g[0] = beta;
      sh.ih = (float)(1.0 / beta);
    });
    if (sh.done != 0) break;
    if (rows_warp) normalise(0);
    gm_barrier(sh, a, buf);   // the product gathers z
    int ku = 0;   // columns of this cycle
    for (int k = 0;; ++k) {
      // (1) w = B z and its dots; meanwhile the scalar warp ends column k - 1
      if (rows_warp) {
        gs_product<KT, !VS>(of, rw, B, z, w, ws, nt);
      } else if (scalar && k > 0) {
        gm_column(sh, k - 1, a, *berr != 0);
      }
      __syncthreads();
      ku = k;
      if (sh.done != 0 || (k > 0 && sh.cycle_done != 0)) break;
      const int R = min(gm_strand_sets(k + 1), S);
      auto value = [&](int q) {
        double t = 0.0;
        for (int r = 0; r < R; ++r) t += sh.fold[q * R + r];
        return t;
      };
      if (rows_warp) gs_dots(sh, rw, w, ws, V, VS, vs, R, S, nwarp, k, true);
      gs_fold(sh, (k + 2) * R);
      // h1 and the DGKS test
      gm_exchange(sh, k + 2, a, buf, value, [&]() {
        const int q = threadIdx.x;
        double h = 0.0;
        if (q <= k) {
          h = sh.tot[q];
          sh.h1[q] = h;
          sh.h2[q] = 0.0;
          sh.hs[q] = (float)h;
        }
        const double ww = sh.tot[k + 1], rest = ww - warp_sum(h * h);
        if (q == 0) sh.skip = rest >= 0.5 * ww && ww > 0.0;
      });
      if (!sh.skip) {   // second projection: w = w - V h1, h2 = V^T w
        if (rows_warp) project(k);
        __syncthreads();
        if (rows_warp) gs_dots(sh, rw, w, ws, V, VS, vs, R, S, nwarp, k, false);
        gs_fold(sh, (k + 1) * R);
        gm_exchange(sh, k + 1, a, buf, value, [&]() {
          const int q = threadIdx.x;
          if (q <= k) {
            const double h = sh.tot[q];
            sh.h2[q] = h;
            sh.hs[q] = (float)h;
          }
        });
      }
      // (2) w -= V h and its norm (meanwhile the scalar warp rotates column k), v_{k+1} = w / ||w||
      if (rows_warp) project(k);
      else gm_rotate(sh, k);
      __syncthreads();
      if (rows_warp) sh.col[threadIdx.x] = gs_norm(rw, w, ws, R, S, nwarp);
      gs_column(sh, nt);
      gm_exchange(sh, 1, a, buf, norm_value, [&]() {
        if (threadIdx.x != 0) return;
        sh.nrm2 = sh.tot[0];
        sh.ih = sh.tot[0] == 0.0 ? 0.f : (float)(1.0 / sqrt(sh.tot[0]));   // 0: the cycle ends with this column
      });
      if (rows_warp) normalise(k + 1);
      gm_barrier(sh, a, buf);
    }
    if (sh.done != 0) break;
    // x += D^{-1} sum_q y_q v_q
    if (threadIdx.x < 32) {
      gm_triangle(sh, ku);
      const int c = threadIdx.x;
      if (c < ku) sh.hs[c] = (float)-sh.y[c];   // the projection's sign
    }
    __syncthreads();
    if (rows_warp) {
#pragma unroll 1
      for (int g = threadIdx.x; g < ng; g += nt) {
        const int l = g * W;
        const int64_t i = rw.at(l);
        const Pack<float> v = gm_project(sh, 0.f, w + (ws ? l : i), V + (VS ? l : i), vs, 0, ku - 1);
#pragma unroll
        for (int e = 0; e < W; ++e)
          if (l + e < rw.nrow) x[i + e] = fma(dinv[i + e], v.e[e], have_x ? x[i + e] : 0.f);
      }
    }
    have_x = true;
    gm_barrier(sh, a, buf);   // the next residual gathers x
  }
  // the solution, and the caller's update unless the solve broke down
  const bool upd = a.ep.u != nullptr && sh.done != 2;
#pragma unroll 1
  for (int l = threadIdx.x; l < rw.nrow; l += blockDim.x) {
    const int64_t i = rw.at(l);
    const double xi = have_x ? (double)x[i] : 0.0;
    a.xout[i] = xi;
    if (upd) krylov_update(a.ep, i, xi);
  }
  if (blockIdx.x == 0 && scalar) gm_report(sh, a, *berr != 0);
}

}  // namespace

void krylov_free(afc_problem_s* p) {
  if (!p->kw) return;
  p->kw->vec.free_();
  p->kw->sc.free_();
  p->kw->part.free_();
  p->kw->barrier.free_();
  pinned_free(p->kw->hsc, kHscBytes);
  delete p->kw;
  p->kw = nullptr;
}

namespace {

// The device must run cooperative launches (GB300 does); its SM count, asked once.
int coop_device(afc_problem_s* p) {
  KrylovWork& w = *p->kw;
  if (w.nsm > 0) return AFC_OK;
  int c = 0;
  AFC_CUDA(cudaDeviceGetAttribute(&c, cudaDevAttrCooperativeLaunch, p->device));
  if (!c) { set_error("the Krylov solvers need a device with cooperative launches"); return AFC_E_CUDA; }
  AFC_CUDA(cudaDeviceGetAttribute(&w.nsm, cudaDevAttrMultiProcessorCount, p->device));
  return AFC_OK;
}

int ensure_work(afc_problem_s* p, int nvec, bool fp32) {
  if (!p->kw) p->kw = new KrylovWork();
  KrylovWork& w = *p->kw;
  const size_t esz = fp32 ? sizeof(float) : sizeof(double);
  const size_t pad = ((size_t)p->pad + 31) & ~(size_t)31;   // vectors start on 16-byte boundaries
  const size_t vstride = (((size_t)p->N + 31) & ~(size_t)31) + 2 * pad;
  const int64_t bytes = (int64_t)(nvec * vstride * esz);
  if (w.vec.base == nullptr || w.vec.n < bytes) {
    if (w.vec.base) AFC_CUDA(cudaStreamSynchronize(p->stream));   // nothing uses the smaller one any more
    int st = w.vec.alloc(bytes);   // zero-filled
    if (st) return st;
  } else if (w.vstride != vstride || w.fp32 != (int)fp32) {
    // halos are read by the SpMV (times zero coefficients): keep them zero
    AFC_CUDA(cudaMemsetAsync(w.vec.base, 0, (size_t)w.vec.n, p->stream));
  }
  w.vstride = vstride;
  w.fp32 = fp32;
  w.N = p->N;
  w.pad = (int)pad;
  if (!w.sc.base) {
    int st = w.sc.alloc(S_END + 8);
    if (st) return st;
    if ((st = w.barrier.alloc(4))) return st;
    if ((st = coop_device(p))) return st;
    if (pinned_alloc((void**)&w.hsc, kHscBytes) != cudaSuccess) {
      set_error("pinned host allocation failed");
      return AFC_E_OOM;
    }
  }
  const int64_t need_part = (int64_t)(kMaxRestart + 4) * std::max<int64_t>(kRedBlocks, grid_for(p->N));
  if (w.part.n < need_part) {
    int st = w.part.alloc(need_part);
    if (st) return st;
  }
  return AFC_OK;
}

template <class T>
T* vec_at(KrylovWork& w, int q) {
  return reinterpret_cast<T*>(w.vec.base) + q * w.vstride + w.pad;
}

// The persistent BiCGStab launch on stream s (no synchronisation).
template <class T>
int bicg_fused_launch(afc_problem_s* p, cudaStream_t s, int system, const T* B, const T* dinv, const afc_opts* o,
                      const double* rhs, double* xout, const KrylovEpilogue* epi) {
  KrylovWork& w = *p->kw;
  int st = coop_device(p);
  if (st) return st;
  const int64_t N = p->N;
  BicgArgs<T> a;
  a.N = N;
  a.sc = w.sc.p;
  a.rhs = rhs;
  a.xout = xout;
  a.loc = vec_at<T>(w, 2);
  a.vstride = w.vstride;
  a.part = w.part.p;
  a.bar = reinterpret_cast<GridBar*>(w.barrier.p);
  a.atol = o->ksp_atol;
  a.rtol = o->ksp_rtol;
  a.maxit = o->ksp_maxit;
  if (epi) a.ep = *epi;
  a.wait_ns = p->grid_wait_ns;
  const int G = (int)std::max<int64_t>(1, std::min<int64_t>((N + 63) / 64, w.nsm));
  const int64_t rows = (N + G - 1) / G;
  const int64_t rounds = (rows + kFusedBlock - 1) / kFusedBlock;
  // A mixed stationary solve amplifies the rounding of its inner solver at isolated nodes (with other
  // sums P1 57^3 moved by up to 6e-10): from several rows a thread on, the sums of its solver have
  // one order, every 512th row of a block to a thread and the partials in turn.  Elsewhere as many
  // threads as share the rows evenly in the fewest rounds, and quarters of the columns (a CN step of
  // Q1 65^3 with single-precision solves is 3 % faster for it).
  const bool turn = sizeof(T) == 4 && system == 0 && rounds > 1;
  const int block = turn ? kFusedBlock : (int)std::max<int64_t>(64, ((rows + rounds - 1) / rounds + 31) / 32 * 32);
  a.rows = (int)rows;
  const size_t local = 6 * (size_t)rows * sizeof(T);
  const bool in_smem = local <= kFusedSmem;
  const size_t smem = in_smem ? local : 0;
  with_K(p->K, [&](auto kc) {
    constexpr int KT = decltype(kc)::value;
    auto kern = in_smem ? k_bicg_fused<KT, T, true, false> : k_bicg_fused<KT, T, false, false>;
    if constexpr (sizeof(T) == 4)
      if (turn) kern = in_smem ? k_bicg_fused<KT, T, true, true> : k_bicg_fused<KT, T, false, true>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kFusedSmem);
    int nb = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, block, smem);
    if (e != cudaSuccess || nb < 1) {
      st = cuda_fail(e != cudaSuccess ? e : cudaErrorInvalidConfiguration, "occupancy of k_bicg_fused");
      return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)G);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaEvent_t ev = prof_start(p);
    e = cudaLaunchKernelEx(&cfg, kern, p->offs, B, dinv, vec_at<T>(w, 0), vec_at<T>(w, 1), a);
    prof_stop(p, "k_bicg_fused", ev);
    if (e != cudaSuccess) st = cuda_fail(e, "cudaLaunchKernelEx(k_bicg_fused)");
  });
  return st;
}

// Host side of a persistent solve just launched: its scalars and status.
int fused_result(afc_problem_s* p, const char* what, int* its, double* res) {
  KrylovWork& w = *p->kw;
  cudaStream_t s = p->stream;
  AFC_CUDA(cudaMemcpyAsync(w.hsc, w.sc.p, S_END * sizeof(double), cudaMemcpyDeviceToHost, s));
  unsigned int* hbar = reinterpret_cast<unsigned int*>(w.hsc + S_END);
  AFC_CUDA(cudaMemcpyAsync(hbar, w.barrier.p, 4 * sizeof(unsigned int), cudaMemcpyDeviceToHost, s));
  AFC_CUDA(cudaStreamSynchronize(s));
  if (its) *its = (int)w.hsc[S_ITS];
  if (res) *res = w.hsc[S_NRES];
  if (hbar[2] != 0u) {
    const int st = krylov_reset_barrier(p);
    if (st) return st;
    set_error(std::string("a grid barrier of the ") + what + " launch gave up waiting");
    return AFC_E_TIMEOUT;
  }
  const double done = w.hsc[S_DONE];
  if (done == 2.0) { set_error(std::string(what) + " breakdown or non-finite value"); return AFC_E_NAN; }
  return done == 1.0 ? AFC_OK : AFC_NOT_CONVERGED;
}

template <class T>
int bicgstab_impl(afc_problem_s* p, int system, const T* B, const T* dinv, const afc_opts* o, const double* rhs, double* xout,
                  int* its, double* res, const KrylovEpilogue* epi) {
  int st = ensure_work(p, kBicgVectors, sizeof(T) == 4);
  if (st) return st;
  if ((st = bicg_fused_launch<T>(p, p->stream, system, B, dinv, o, rhs, xout, epi))) return st;
  return fused_result(p, "BiCGStab", its, res);
}

// The persistent GMRES launch on stream s (no synchronisation).  One block per SM at most.  In
// double small systems spread over all SMs, 64 rows a block, because a block's FP64 sums cost
// 16 cycles per warp.  In single precision a block takes two chunks (512 rows) where there are SMs
// enough: solves on other streams find room beside it, at no cost to a solve alone (measured with
// at least 512 rows a block against 64: a burst of 8 served requests 108 -> 76 ms, P1 17^3 to Q1 33^3
// within 1 %).
template <class T>
int gmres_fused_launch(afc_problem_s* p, cudaStream_t s, const T* B, const T* dinv, const afc_opts* o,
                       const double* rhs, double* xout, const KrylovEpilogue* epi) {
  KrylovWork& w = *p->kw;
  int st = AFC_OK;
  const int64_t N = p->N;
  GmArgs a;
  a.N = N;
  a.sc = w.sc.p;
  a.rhs = rhs;
  a.xout = xout;
  a.vstride = w.vstride;
  a.bar = reinterpret_cast<GridBar*>(w.barrier.p);
  a.part = w.part.p;
  a.atol = o->ksp_atol;
  a.rtol = o->ksp_rtol;
  a.maxit = o->ksp_maxit;
  a.m = o->gmres_restart;
  if (epi) a.ep = *epi;
  a.wait_ns = kBarrierWaitNs;   // afc_set_grid_wait_limit is of the BiCGStab launches
  constexpr bool kSingle = sizeof(T) == 4;
  const int64_t unit = kSingle ? kGsChunk : kGmUnit, units = (N + unit - 1) / unit;
  const int64_t least = kSingle ? 2 : 64 / kGmUnit;   // units of a block, at least
  const int G = (int)std::max<int64_t>(1, std::min<int64_t>((units + least - 1) / least, std::min(w.nsm, 160)));
  const int64_t rows = (units + G - 1) / G * unit;   // most rows of a block
  const size_t vec = (size_t)rows * sizeof(T);
  const bool vs = (size_t)(a.m + 2) * vec <= kGmSmem;   // w and V_0 .. V_m
  a.w_in_smem = vec <= kGmSmem;
  a.rows = (int)rows;
  const size_t smem = vs ? (a.m + 2) * vec : a.w_in_smem ? vec : 0;
  const int most = (vs ? kGmBlockS : kGmBlock) - 32;
  a.compute = (int)std::max<int64_t>(kGmMinCompute, std::min<int64_t>(most, (rows + 31) / 32 * 32));
  const int block = a.compute + 32;
  with_K(p->K, [&](auto kc) {
    constexpr int KT = decltype(kc)::value;
    auto kern = [&] {
      if constexpr (kSingle) return vs ? k_gm_single<KT, true> : k_gm_single<KT, false>;
      else return vs ? k_gm_fused<KT, T, true> : k_gm_fused<KT, T, false>;
    }();
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kGmSmem);
    int nb = 0;
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kern, block, smem);
    if (e != cudaSuccess || nb < 1) {
      st = cuda_fail(e != cudaSuccess ? e : cudaErrorInvalidConfiguration, "occupancy of the GMRES launch");
      return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)G);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaEvent_t ev = prof_start(p);
    e = cudaLaunchKernelEx(&cfg, kern, p->offs, B, dinv, vec_at<T>(w, 0), vec_at<T>(w, 1), vec_at<T>(w, 2),
                           vec_at<T>(w, 3), a);
    prof_stop(p, kSingle ? "k_gm_single" : "k_gm_fused", ev);
    if (e != cudaSuccess) st = cuda_fail(e, "cudaLaunchKernelEx(GMRES)");
  });
  return st;
}

int gmres_work(afc_problem_s* p, const afc_opts* o, bool fp32) {
  const int m = o->gmres_restart;
  if (m < 1 || m > kMaxRestart) { set_error("gmres_restart must be in 1..32"); return AFC_E_INVALID; }
  return ensure_work(p, 3 + m + 1, fp32);   // x, z, w, V_0 .. V_m
}

template <class T>
int gmres_impl(afc_problem_s* p, const T* B, const T* dinv, const afc_opts* o, const double* rhs, double* xout,
               int* its, double* res, const KrylovEpilogue* epi) {
  int st = gmres_work(p, o, sizeof(T) == 4);
  if (st) return st;
  if ((st = gmres_fused_launch<T>(p, p->stream, B, dinv, o, rhs, xout, epi))) return st;
  return fused_result(p, "GMRES", its, res);
}

}  // namespace

namespace {

template <class T>
int bicgstab_graph(afc_problem_s* p, int system, const T* B, const T* dinv, const afc_opts* o, const double* rhs, double* xout,
                   cudaStream_t cs, cudaGraph_t g, std::vector<cudaGraphNode_t>& frontier, const KrylovEpilogue* epi) {
  int st = ensure_work(p, kBicgVectors, sizeof(T) == 4);
  if (st) return st;
  return capture_into(p, cs, g, frontier, [&]() -> int {
    return bicg_fused_launch<T>(p, p->stream, system, B, dinv, o, rhs, xout, epi);
  }, frontier);
}

template <class T>
int gmres_graph(afc_problem_s* p, const T* B, const T* dinv, const afc_opts* o, const double* rhs, double* xout,
                cudaStream_t cs, cudaGraph_t g, std::vector<cudaGraphNode_t>& frontier, const KrylovEpilogue* epi) {
  int st = gmres_work(p, o, sizeof(T) == 4);
  if (st) return st;
  return capture_into(p, cs, g, frontier, [&]() -> int {
    return gmres_fused_launch<T>(p, p->stream, B, dinv, o, rhs, xout, epi);
  }, frontier);
}

}  // namespace

int krylov_prepare(afc_problem_s* p, const afc_opts* o) {
  const bool fp32 = o->precision == AFC_MIXED;
  if (fp32 && p->precision != AFC_MIXED) {
    set_error("mixed-precision solve needs afc_assemble(..., AFC_MIXED)");
    return AFC_E_STATE;
  }
  return o->ksp == AFC_KSP_GMRES ? gmres_work(p, o, fp32) : ensure_work(p, kBicgVectors, fp32);
}

int krylov_graph(afc_problem_s* p, int system, const afc_opts* o, const double* rhs, double* x, cudaStream_t cs,
                 cudaGraph_t g, std::vector<cudaGraphNode_t>& frontier, const KrylovEpilogue* epi) {
  const bool gm = o->ksp == AFC_KSP_GMRES;
  if (o->precision == AFC_MIXED) {
    const float* B = system == 0 ? p->Bst32.p : p->Bcn32.p;
    const float* di = system == 0 ? p->dinv_st32.p : p->dinv_cn32.p;
    return gm ? gmres_graph<float>(p, B, di, o, rhs, x, cs, g, frontier, epi)
              : bicgstab_graph<float>(p, system, B, di, o, rhs, x, cs, g, frontier, epi);
  }
  const double* B = system == 0 ? p->Bst.p : p->Bcn.p;
  const double* di = system == 0 ? p->dinv_st.p : p->dinv_cn.p;
  return gm ? gmres_graph<double>(p, B, di, o, rhs, x, cs, g, frontier, epi)
            : bicgstab_graph<double>(p, system, B, di, o, rhs, x, cs, g, frontier, epi);
}

int krylov_reset_barrier(afc_problem_s* p) {
  if (!p->kw || !p->kw->barrier.p) return AFC_OK;
  AFC_CUDA(cudaMemsetAsync(p->kw->barrier.p, 0, 4 * sizeof(unsigned int), p->stream));
  AFC_CUDA(cudaStreamSynchronize(p->stream));
  return AFC_OK;
}
const void* krylov_key(afc_problem_s* p) { return p->kw ? (const void*)p->kw->vec.base : nullptr; }

int krylov_solve(afc_problem_s* p, int system, const afc_opts* o, const double* rhs, double* x, int* its,
                 double* res, const KrylovEpilogue* epi) {
  const bool mixed = o->precision == AFC_MIXED;
  if (mixed && p->precision != AFC_MIXED) {
    set_error("mixed-precision solve needs afc_assemble(..., AFC_MIXED)");
    return AFC_E_STATE;
  }
  if (system == 1 && p->cn_dt < 0.0) { set_error("CN system not built"); return AFC_E_STATE; }
  const bool gm = o->ksp == AFC_KSP_GMRES;
  if (mixed) {
    const float* B = system == 0 ? p->Bst32.p : p->Bcn32.p;
    const float* di = system == 0 ? p->dinv_st32.p : p->dinv_cn32.p;
    return gm ? gmres_impl<float>(p, B, di, o, rhs, x, its, res, epi)
              : bicgstab_impl<float>(p, system, B, di, o, rhs, x, its, res, epi);
  }
  const double* B = system == 0 ? p->Bst.p : p->Bcn.p;
  const double* di = system == 0 ? p->dinv_st.p : p->dinv_cn.p;
  return gm ? gmres_impl<double>(p, B, di, o, rhs, x, its, res, epi)
            : bicgstab_impl<double>(p, system, B, di, o, rhs, x, its, res, epi);
}

}  // namespace afc
