// Per-row arithmetic of the explicit FE-SSP stage with Zalesak's limiter
// (Sec. 2.1.2, Sec. 2.1.3), shared by the one-problem kernels (fct.cu) and the
// batched kernels (batch.cu) so that an instance gives the same bits alone and
// in a batch.
//
// The stage has four passes, each needing the previous one on the neighbours:
//   rate     y = AA u, udot^L = (f - y) / m, predictor u~ = u + dt udot^L
//   edges    r_ij of every pair, once per pair at its lower row (Eq. defn_r_ij_SSP)
//   factors  P+/-, Q+/- over N_i, R+/- (Zalesak steps 1-3); in its FUSED form it also forms the
//            fluxes, both ends each (r_ji = -r_ij bit for bit: every rounding is symmetric),
//            and stores the upper ones, so that the edges pass is not needed
//   correct  alpha_ij, F*_i = sum_j alpha_ij r_ij, u_new = u~ + dt F* / m, and the
//            SSP combination out = a uA + b u_new
//
// Mixed precision (MIXED = true): the raw flux r_ij of a pair is formed in single
// precision, from single-precision copies of m_ij, d_ij, u and udot^L, and stored
// as a float; P+/-, Q+/-, R+/-, alpha, F* and the lumped-mass update stay in
// double and use the float fluxes widened exactly, so the limiter's local bounds
// hold for the fluxes that are actually applied.
#pragma once

#include "kernels_common.cuh"

namespace afc {

// Pointers of one instance for the stage passes.  Node vectors carry the halo.
// No pointer here or in the row functions is __restrict__: a persistent batched
// launch writes, in one pass, arrays that later passes of the same launch read,
// so their loads must not take the read-only (non-coherent) cache path.
struct SspArrays {
  int64_t N;
  const double* AA;                 // K * N low-order operator
  const double* m_up;               // Kup * N
  const double* d_up;               // Kup * N
  const float2* md32;               // Kup * N (mixed): (m_ij, d_ij)
  const double* mL;
  const double* imL;                // 1 / m_i
  const double* f;
  const uint8_t* dir;
  const double* udir;
  const unsigned long long* mask;
  double* udot;
  double* ut;
  float2* uw;                       // mixed: (u, udot^L) rounded to single (halo)
  double* r_up;                     // Kup * N
  float* r32;                       // Kup * N (mixed)
  double* Rp;                       // halo
  double* Rm;
  double* Fs;                       // F* of the stage (may be null)
};

// rate pass at row i (udot^L = 0 at Dirichlet nodes, whose data is constant in time)
template <int KT, bool MIXED>
__device__ __forceinline__ void ssp_rate_row(const Offsets& of, const SspArrays& a, int64_t i,
                                             const double* u, double dt) {
  const int K = KT > 0 ? KT : of.K;
  const int64_t N = a.N;
  double y = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) y = fma(a.AA[k * N + i], u[i + of.o[k]], y);
  const double ui = u[i];
  double ud, uti;
  if (a.dir[i]) {
    ud = 0.0;
    uti = a.udir[i];
  } else {
    ud = div_by(a.f[i] - y, a.mL[i], a.imL[i]);
    uti = fma(dt, ud, ui);
  }
  a.ut[i] = uti;
  if (MIXED) a.uw[i] = make_float2(__double2float_rn(ui), __double2float_rn(ud));
  else a.udot[i] = ud;
}

// r_ij = m_ij (udot_i - udot_j) + d_ij (u_j - u_i); w = (u, udot), c = (m_ij, d_ij)
__device__ __forceinline__ float ssp_flux(float2 c, float2 wi, float2 wj) {
  return fmaf(c.x, wi.y - wj.y, c.y * (wj.x - wi.x));
}

// edges pass: the Kup pairs (i, i + o) with o > 0 stored at row i
template <int KT, bool MIXED>
__device__ __forceinline__ void ssp_edges_row(const Offsets& of, const SspArrays& a, int64_t i,
                                              const double* u) {
  const int Kup = (KT > 0 ? KT : of.K) / 2;
  const int64_t N = a.N;
  if (MIXED) {
    const float2 wi = a.uw[i];
#pragma unroll
    for (int ku = 0; ku < Kup; ++ku) {
      const int64_t q = (int64_t)ku * N + i;
      a.r32[q] = ssp_flux(a.md32[q], wi, a.uw[i + of.o[Kup + 1 + ku]]);
    }
  } else {
    const double ui = u[i], udi = a.udot[i];
#pragma unroll
    for (int ku = 0; ku < Kup; ++ku) {
      const int64_t q = (int64_t)ku * N + i;
      const int64_t j = i + of.o[Kup + 1 + ku];
      a.r_up[q] = fma(a.m_up[q], udi - a.udot[j], a.d_up[q] * (u[j] - ui));
    }
  }
}

// factors pass: P+/- from the stored fluxes, Q+/- from the predictor over N_i, R+/-
// (FUSED: mixed only)
template <int KT, bool MIXED, bool FUSED, int S = kGroup<KT>, bool SMALL = false>
__device__ __forceinline__ void ssp_factors_row(const Offsets& of, const SspArrays& a, int64_t i, const double* u,
                                                double dt) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  // SMALL: the row's own data before the test of its Dirichlet flag (one wait, not two)
  unsigned long long mk = SMALL ? a.mask[i] : 0ull;
  double uti = SMALL ? a.ut[i] : 0.0, m = SMALL ? a.mL[i] : 0.0;
  const bool isdir = a.dir[i];
  if (isdir) {
    a.Rp[i] = 1.0;
    a.Rm[i] = 1.0;
    if (!FUSED) return;
  }
  if (FUSED && isdir) {   // its upper fluxes all the same: their other ends read them
    ssp_edges_row<KT, MIXED>(of, a, i, u);
    return;
  }
  if (!SMALL) {
    mk = a.mask[i];
    uti = a.ut[i];
  }
  // P+/- on the integer pipe (one rounding at the end), one flux at a time: two FP64 adds per
  // pair took 52 of the pass's 82 FP64 warp instructions at Q1, and holding a row's fluxes
  // until their largest exponent is known took it to 48 registers
  SignedSums64 acc;
  long long kmax = dkey(uti), kmin = kmax;
#pragma unroll
  for (int k0 = 0; k0 < K; k0 += S) {
    double r[S], v[S];
    float rf[S];
    if (FUSED) {
      float2 c[S], w[S];
      const float2 wi = a.uw[i];
#pragma unroll
      for (int j = 0; j < S; ++j) {
        if (k0 + j == Kup) continue;
        const int k = group_at<KT>(k0 + j, K);
        c[j] = a.md32[pair_slot(of, Kup, k, i, a.N)];
        w[j] = a.uw[i + of.o[k]];
        v[j] = a.ut[i + of.o[k]];
      }
#pragma unroll
      for (int j = 0; j < S; ++j) {
        if (k0 + j == Kup) continue;
        // upper pairs as the edges pass stores them; lower ones as their lower row does, r_e = -r_ij
        rf[j] = k0 + j > Kup ? ssp_flux(c[j], wi, w[j]) : ssp_flux(c[j], w[j], wi);
        if (k0 + j > Kup) a.r32[(int64_t)(group_at<KT>(k0 + j, K) - Kup - 1) * a.N + i] = rf[j];
      }
    } else {
#pragma unroll
      for (int j = 0; j < S; ++j) {
        if (k0 + j == Kup) continue;
        const int k = group_at<KT>(k0 + j, K);
        const int64_t q = pair_slot(of, Kup, k, i, a.N);
        if (MIXED) rf[j] = a.r32[q];
        else r[j] = a.r_up[q];
        v[j] = a.ut[i + of.o[k]];
      }
    }
#pragma unroll
    for (int j = 0; j < S; ++j) {
      const int k = k0 + j;
      if (k == Kup || !((mk >> k) & 1ull)) continue;
      if (MIXED) acc.add(__float_as_uint(rf[j]) ^ (k > Kup ? 0u : 0x80000000u));   // r_ij = -r_ji
      else acc.add((unsigned long long)__double_as_longlong(r[j]) ^ (k > Kup ? 0ull : 0x8000000000000000ull));
      const long long kj = dkey(v[j]);
      kmax = kj > kmax ? kj : kmax;
      kmin = kj < kmin ? kj : kmin;
    }
  }
  double Pp, Pm;
  acc.result<MIXED ? 127 : 1023>(Pp, Pm);
  // A NaN flux of the row comes from a rate that is NaN, and so is a predictor of N_i (its key lies
  // beyond those of the infinities): the totals it is in are then NaN as FP64 adds would leave them.
  // (Seen at each value it cost 5 % of a step of 2.1 M rows.)
  if (!MIXED && (kmax > 0x7ff0000000000000ll || kmin < (long long)0x800fffffffffffffull)) {
    const long long inf = 0x7ff0000000000000ll, nan = 0x7ff8000000000000ll;
    if (__double_as_longlong(Pp) == inf) Pp = __longlong_as_double(nan);
    if (__double_as_longlong(neg_bits(Pm)) == inf) Pm = neg_bits(__longlong_as_double(nan));
  }
  // >= 0 and <= 0: the max / min include i itself
  const double Qp = from_key(kmax) - uti, Qm = from_key(kmin) - uti;
  if (!SMALL) m = a.mL[i];
  a.Rp[i] = zalesak_factor(m * Qp, dt * Pp);
  a.Rm[i] = zalesak_factor(m * Qm, dt * Pm);
}

// A load that stays where it is written (the compiler would move it behind the test that picks
// one of two, and so behind the wait for the flux).
__device__ __forceinline__ double load_now(const double* p) {
  double v;
  asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return v;
}

// correct pass and the SSP combination; returns the new value written to out[i]
// SMALL (grids that do not fill the GPU) also loads both factors of every neighbour beside its
// flux, one wait for memory per group (12.5 us against 16.4 us for 77,121 rows of Q1, mixed),
// instead of the one that the flux's sign asks for, half the loads (143 us against 200 us for
// 2.1 M rows).
template <int KT, bool MIXED, int S = kGroup<KT>, bool SMALL = false>
__device__ __forceinline__ void ssp_correct_row(const Offsets& of, const SspArrays& a, int64_t i, int limiter,
                                                double dt, double ca, const double* uA, double cb,
                                                double* out) {
  const int K = KT > 0 ? KT : of.K, Kup = K / 2;
  double unew;
  double F = 0.0;
  unsigned long long mk = SMALL ? a.mask[i] : 0ull;
  double ut = 0.0, m = 0.0, im = 0.0, ua = 0.0;
  if (SMALL) {   // the row's own data before the test of its Dirichlet flag
    ut = a.ut[i];
    m = a.mL[i];
    im = a.imL[i];
    if (ca != 0.0) ua = uA[i];
  }
  if (a.dir[i]) {
    unew = a.udir[i];
  } else {
    if (limiter != AFC_LIM_NONE) {
      if (!SMALL) mk = a.mask[i];
      const double rpi = a.Rp[i], rmi = a.Rm[i];
#pragma unroll
      for (int k0 = 0; k0 < K; k0 += S) {
        double r[S], Rj[S], Rk[S];
        // single-precision fluxes are widened after the group's loads: the widening's test for
        // subnormals is a branch that each following load waited behind (mixed SSP3 step of Q1 41x33x57
        // 114.7 -> 104.6 us, 97^3 685 -> 614 us; 15 passes over 48 batched instances 7.98 -> 7.60 ms; a
        // widening without a branch, every lane taking the longer way: 107, 664 us and 8.2 ms)
        float rf[S];
#pragma unroll
        for (int j = 0; j < S; ++j) {
          if (k0 + j == Kup) continue;
          const int k = group_at<KT>(k0 + j, K);
          const int64_t q = pair_slot(of, Kup, k, i, a.N);
          if (MIXED) rf[j] = a.r32[q];
          else r[j] = a.r_up[q];
          if (SMALL && limiter == AFC_LIM_ZALESAK) {
            Rj[j] = load_now(a.Rm + i + of.o[k]);
            Rk[j] = load_now(a.Rp + i + of.o[k]);
          }
        }
#pragma unroll
        for (int j = 0; j < S; ++j) {
          if (k0 + j == Kup) continue;
          if (MIXED) r[j] = widen_exact(rf[j]);
          if (k0 + j < Kup) r[j] = neg_bits(r[j]);
        }
        if (!SMALL && limiter == AFC_LIM_ZALESAK) {
#pragma unroll
          for (int j = 0; j < S; ++j)
            if (k0 + j != Kup) Rj[j] = Rk[j] = (gt0(r[j]) ? a.Rm : a.Rp)[i + of.o[group_at<KT>(k0 + j, K)]];
        }
#pragma unroll
        for (int j = 0; j < S; ++j) {
          const int k = k0 + j;
          if (k == Kup || !((mk >> k) & 1ull)) continue;
          if (limiter == AFC_LIM_ZALESAK) F = fma(gt0(r[j]) ? imin_nn(rpi, Rj[j]) : imin_nn(rmi, Rk[j]), r[j], F);
          else F += r[j];
        }
      }
    }
    if (!SMALL) {
      ut = a.ut[i];
      m = a.mL[i];
      im = a.imL[i];
    }
    unew = ut + div_by(dt * F, m, im);
  }
  if (a.Fs) a.Fs[i] = F;
  if (!SMALL && ca != 0.0) ua = uA[i];
  out[i] = ca != 0.0 ? ca * ua + cb * unew : cb * unew;
}

}  // namespace afc
