// Small device helpers shared by the hot-path kernels.
#pragma once

#include <climits>
#include <cmath>
#include <type_traits>

#include "afc_internal.h"

namespace afc {

// m_ij and d_ij of the pair (i, i + o_k), k != Kup.  Stored once per pair at the
// row of the pair's lower node, offset index ku of the positive offset |o_k|.
__device__ __forceinline__ void pair_coef(const Offsets& of, int k, int64_t i, int64_t N,
                                          const double* __restrict__ m_up, const double* __restrict__ d_up,
                                          double& m, double& d) {
  int64_t q;
  if (k > of.Kup) q = (int64_t)(k - of.Kup - 1) * N + i;
  else q = (int64_t)(of.Kup - 1 - k) * N + i + of.o[k];
  m = m_up[q];
  d = d_up[q];
}

__device__ __forceinline__ double pair_d(const Offsets& of, int k, int64_t i, int64_t N,
                                         const double* __restrict__ d_up) {
  if (k > of.Kup) return d_up[(int64_t)(k - of.Kup - 1) * N + i];
  return d_up[(int64_t)(of.Kup - 1 - k) * N + i + of.o[k]];
}

// ---- comparisons on the integer pipe ----------------------------------------
// GB300 runs FP64 compares, min/max and arithmetic on a pipe that issues 2 thread
// operations per SM and cycle.  Comparisons of finite doubles are done here on
// their bit patterns instead: key() maps a double to an int64 with the same
// order (-0 sorts just below +0), so every decision below is exact.
__device__ __forceinline__ long long dkey(double x) {
  const long long b = __double_as_longlong(x);
  return b ^ ((b >> 63) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ bool gt0(double x) { return __double_as_longlong(x) > 0; }      // x > 0
__device__ __forceinline__ bool lt0(double x) { return dkey(x) < -1; }                      // x < 0
__device__ __forceinline__ bool is0(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ double imin(double a, double b) { return dkey(a) <= dkey(b) ? a : b; }
__device__ __forceinline__ double imax(double a, double b) { return dkey(a) >= dkey(b) ? a : b; }
// keys are their own inverse: key(key(x)) = x
__device__ __forceinline__ double from_key(long long k) {
  return __longlong_as_double(k ^ ((k >> 63) & 0x7fffffffffffffffLL));
}
__device__ __forceinline__ double abs_bits(double x) {
  return __longlong_as_double(__double_as_longlong(x) & 0x7fffffffffffffffLL);
}
__device__ __forceinline__ double neg_bits(double x) {
  return __longlong_as_double(__double_as_longlong(x) ^ (long long)0x8000000000000000ULL);
}

// Exact float -> double on the integer pipe (every user of a flux widens it the same
// way, so P+/- and F* see the same values).  A subnormal float m * 2^-149 becomes the
// normal double 2^(p - 149) (m / 2^p), p the position of m's leading bit.
__device__ __forceinline__ double widen_exact(float x) {
  const unsigned b = __float_as_uint(x);
  const unsigned e = (b >> 23) & 0xffu, m = b & 0x7fffffu;
  const unsigned long long s = (unsigned long long)(b & 0x80000000u) << 32;
  if (e == 0u) {
    if (m == 0u) return __longlong_as_double((long long)s);
    const unsigned p = 31u - (unsigned)__clz(m);   // 0 .. 22
    return __longlong_as_double(
        (long long)(s | ((unsigned long long)(p + 874u) << 52) | ((unsigned long long)(m ^ (1u << p)) << (52u - p))));
  }
  const unsigned long long de = e == 0xffu ? 0x7ffull : (unsigned long long)(e + 896u);
  return __longlong_as_double((long long)(s | (de << 52) | ((unsigned long long)m << 29)));
}

// Sums of the positive and of the negative values of a row's pair fluxes in 64-bit fixed point
// (Zalesak's P+ and P-), on the integer pipe.  Each of the two has a scale of its own: its largest
// value's leading bit at bit 57 (up to 62 terms fit), every other term, and the total when a larger
// one rescales it, rounded to the last bit; the totals are rounded to double once.  A total of n
// terms so carries at most 2 n 2^-58 of its own largest term and one rounding, where a sum of FP64
// adds carries n - 1 roundings.  (With one scale for both, a P- below 2^-58 of P+ came out as 0,
// and R- as 1.)  Subnormal values keep their bits.
// On GB300 this replaces two FP64 adds per value (an FP64 warp instruction occupies the pipe for
// 16 cycles).  The values are taken one at a time, so that none has to be kept until the largest
// exponent is known.
struct SignedSums64 {
  unsigned ep = 0u, en = 0u;
  unsigned long long p = 0ull, n = 0ull;

  // m: the significand, a normal value's leading bit at bit 58; e >= 1
  __device__ __forceinline__ void put(unsigned long long m, unsigned e, bool neg) {
    unsigned at = neg ? en : ep;
    unsigned long long t = neg ? n : p;
    if (e > at) {   // scale the total to the larger exponent
      const unsigned d = e - at;
      t = d < 64u ? ((t >> (d - 1u)) + 1ull) >> 1 : 0ull;
      at = e;
    }
    const unsigned sh = at - e;
    t += ((sh < 64u ? m >> sh : 0ull) + 1ull) >> 1;
    if (neg) {
      en = at;
      n = t;
    } else {
      ep = at;
      p = t;
    }
  }
  __device__ __forceinline__ void add(unsigned long long b) {   // a double
    if ((b << 1) == 0ull) return;
    const unsigned e = (unsigned)(b >> 52) & 0x7ffu;
    const unsigned long long f = b & 0xFFFFFFFFFFFFFull;
    put((e ? f | 0x10000000000000ull : f) << 6, e ? e : 1u, b >> 63);
  }
  __device__ __forceinline__ void add(unsigned b) {   // a float
    if ((b << 1) == 0u) return;
    const unsigned e = (b >> 23) & 0xffu, f = b & 0x7fffffu;
    put((unsigned long long)(e ? f | 0x800000u : f) << 35, e ? e : 1u, b >> 31);
  }
  // totals of doubles (BIAS 1023) or floats (BIAS 127)
  template <int BIAS>
  __device__ __forceinline__ void result(double& pos, double& neg) const {
    pos = to_double(p, (int)ep - BIAS - 57);
    neg = neg_bits(to_double(n, (int)en - BIAS - 57));
  }
  __device__ static __noinline__ double to_double_edge(unsigned long long v, int ex) {
    return scalbn(__ull2double_rn(v), ex);
  }
  __device__ static __forceinline__ double to_double(unsigned long long v, int ex) {
    if (v == 0ull) return 0.0;
    const long long d = __double_as_longlong(__ull2double_rn(v));
    const int be = (int)(d >> 52) + ex;
    if (be <= 0 || be >= 2047) return to_double_edge(v, ex);
    return __longlong_as_double(d + ((long long)ex << 52));
  }
};

// The same sums with 64 bits more (the CN scheme's, whose factors enter every correction of a
// step's fixed point): what falls off the end is below 2^-120 of a sum's largest term, and each
// total is rounded to double once.
struct SignedSums128 {
  unsigned ep = 0u, en = 0u;
  unsigned long long ph = 0ull, pl = 0ull, nh = 0ull, nl = 0ull;   // largest term's leading bit: bit 57 of the high word

  __device__ __forceinline__ void add(unsigned long long b) {   // a double
    if ((b << 1) == 0ull) return;
    unsigned e = (unsigned)(b >> 52) & 0x7ffu;
    unsigned long long m = b & 0xFFFFFFFFFFFFFull;
    if (e) m |= 0x10000000000000ull;
    else e = 1u;
    m <<= 5;
    const bool neg = b >> 63;
    unsigned at = neg ? en : ep;
    unsigned long long h = neg ? nh : ph, l = neg ? nl : pl;
    if (e > at) {   // scale the total to the larger exponent
      shift(h, l, e - at);
      at = e;
    }
    unsigned long long vl = 0ull;
    shift(m, vl, at - e);
    l += vl;
    h += m + (l < vl ? 1ull : 0ull);
    if (neg) {
      en = at;
      nh = h;
      nl = l;
    } else {
      ep = at;
      ph = h;
      pl = l;
    }
  }
  __device__ static __forceinline__ void shift(unsigned long long& h, unsigned long long& l, unsigned d) {   // right
    if (d == 0u) return;
    if (d < 64u) {
      l = (l >> d) | (h << (64u - d));
      h >>= d;
    } else {
      l = d < 128u ? h >> (d - 64u) : 0ull;
      h = 0ull;
    }
  }
  // A total whose largest term is normal has its leading bit at bit 57 of the high word or above, so
  // that the low word matters to the rounding only by being zero or not; one of subnormal terms is
  // exact in the high word.
  __device__ __forceinline__ void result(double& pos, double& neg) const {
    pos = SignedSums64::to_double(ph | (pl != 0ull ? 1ull : 0ull), (int)ep - 1023 - 57);
    neg = neg_bits(SignedSums64::to_double(nh | (nl != 0ull ? 1ull : 0ull), (int)en - 1023 - 57));
  }
};

// a / m for a divisor whose rounded reciprocal im is at hand (Markstein, IBM J. Res. Dev. 34
// (1990) 111): q = a im, one residual, one correction, three FP64 operations where the inlined
// division takes about ten; the correctly rounded quotient, as long as nothing in it
// under- or overflows.  A product that is not finite is returned as it is.
__device__ __forceinline__ double div_by(double a, double m, double im) {
  const double q = a * im;
  const double c = fma(fma(-q, m, a), im, q);
  return (__double_as_longlong(q) & 0x7ff0000000000000ll) == 0x7ff0000000000000ll ? q : c;
}

// min / max of two values known to be >= 0 (correction factors, bounds): plain int compare
__device__ __forceinline__ double imin_nn(double a, double b) {
  return __double_as_longlong(a) <= __double_as_longlong(b) ? a : b;
}
// Exact 0.5 * x (IEEE, ties to even) on the integer pipe.  Normal numbers above the
// smallest binade move their exponent; zeros, subnormals and the smallest binade
// halve the 53-bit significand with round-half-even; Inf and NaN pass through.  No
// branch issues an FP64 instruction, so none costs the FP64 pipe even when the
// compiler evaluates both sides of a branch.
__device__ __forceinline__ double half_exact(double x) {
  const long long b = __double_as_longlong(x);
  const long long e = (b >> 52) & 0x7ff;
  if (e > 1 && e < 0x7ff) return __longlong_as_double(b - (1LL << 52));
  if (e == 0x7ff) return x;
  const long long sign = b & (long long)0x8000000000000000ULL;
  const unsigned long long M = (unsigned long long)(b & 0x000FFFFFFFFFFFFFLL) | (e == 1 ? (1ULL << 52) : 0ULL);
  unsigned long long h = M >> 1;
  if ((M & 1ULL) && (h & 1ULL)) ++h;   // exactly half-way: to even (may carry into the exponent)
  return __longlong_as_double(sign | (long long)h);
}

// R = min{1, num / den} of Zalesak's step 3 for num = m_i Q, den = dt P of the same sign,
// R = 1 if P = 0.  For same-sign num, den the rounded quotient reaches 1 exactly when
// |num| >= |den|, so the division is only done where R < 1 (same result bit for bit).
__device__ __forceinline__ double zalesak_factor(double num, double den) {
  if (is0(den)) return 1.0;
  const long long an = __double_as_longlong(num) & 0x7fffffffffffffffLL;
  const long long ad = __double_as_longlong(den) & 0x7fffffffffffffffLL;
  if (an >= ad) return 1.0;
  return num / den;
}

// minmod of Eq. prelimiting: 0 unless both arguments have the same strict sign.
__device__ __forceinline__ double minmod(double a, double b) {
  if (gt0(a) && gt0(b)) return imin(a, b);
  if (lt0(a) && lt0(b)) return imax(a, b);
  return 0.0;
}

// The antidiffusive flux of the pair (i, i + o_k) seen from row i, for a flux
// stored once per pair at the pair's lower row: r_ij = r_e (k > Kup) or -r_e.
__device__ __forceinline__ double pair_flux(const Offsets& of, int Kup, int k, int64_t i, int64_t N,
                                            const double* __restrict__ r_up) {
  if (k > Kup) return r_up[(int64_t)(k - Kup - 1) * N + i];
  return neg_bits(r_up[(int64_t)(Kup - 1 - k) * N + i + of.o[k]]);   // -r_e, sign bit on the integer pipe
}

// Index of the pair (i, i + o_k) in pair data stored at the pair's lower row, for loads that
// are issued whether or not the pair is in the pattern (the caller drops the value of an
// absent one): always inside the array.  (A pair below the first row would start before it.)
__device__ __forceinline__ int64_t pair_slot(const Offsets& of, int Kup, int k, int64_t i, int64_t N) {
  if (k > Kup) return (int64_t)(k - Kup - 1) * N + i;
  const int64_t q = (int64_t)(Kup - 1 - k) * N + i + of.o[k];
  return q < 0 ? 0 : q;
}
// Neighbours whose loads a row issues together: a third of the structured patterns (a loop
// that tests the pattern before each load waits for one load after the other, 12 us for a
// pass over 729 rows; all at once take the registers of two rows).  Other patterns take three at a
// time (one at a time: SSP3 step of 3,689 nodes with 45 offsets 171 us, now 137, batched 189, now 159); their last group
// may reach past the pattern and loads its last offset again (group_at), which the row's mask drops:
// 3 divides kMaxOffsets, so that the group stays within 63 offsets.
template <int KT>
constexpr int kGroup = KT == 27 ? 9 : KT == 15 ? 5 : 3;
static_assert(kMaxOffsets % 3 == 0, "the last group of a pattern of any size");
template <int KT>
__device__ __forceinline__ int group_at(int k, int K) {
  return KT > 0 || k < K ? k : K - 1;
}

template <class T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Block sums in a fixed order.  On GB300 every FP64 warp instruction costs the
// FP64 pipe 16 cycles whatever its active lanes, so a shuffle tree in every warp
// (5 adds per warp) is the expensive way to sum a block.  Instead every thread
// stores its value in shared memory and warp 0 alone sums them: each lane adds
// blockDim/32 values, then one shuffle tree (blockDim/32 - 1 + 5 adds per block
// instead of 5 per warp).  Blocks of more than kBlock threads take the shuffle
// route.  Every thread of the block must call these.
__device__ __forceinline__ double warp0_column_sum(const double* col) {
  const int lane = threadIdx.x;   // < 32
  double t = col[lane];
  for (int w = lane + 32; w < (int)blockDim.x; w += 32) t += col[w];
  return warp_sum(t);
}

// The final sum over a pass's block partials, in an order that does not depend on the size of
// the block that forms it (at least one full warp): eight strands, strand w adding partials
// 32 w + lane, then + 256, ... four at a time and then its lanes, one warp per strand in turn;
// the strands are added in pairs.  The fixed point's stop test in the solvers and the host-
// driven loop (k_finalize_sum) so see the same bits.  The loads go through L2.  Every thread
// of the block calls it and receives the total.
__device__ __forceinline__ double final_sum(const double* part, int n) {
  __shared__ double strand[8];
  const int lane = threadIdx.x & 31;
  for (int w = threadIdx.x >> 5; w < 8; w += blockDim.x >> 5) {
    double v = 0.0;
    for (int q = 32 * w + lane; q - lane < n; q += 1024) {
      double x[4];
#pragma unroll
      for (int m = 0; m < 4; ++m) x[m] = q + 256 * m < n ? __ldcg(part + q + 256 * m) : 0.0;
      v += (x[0] + x[1]) + (x[2] + x[3]);
    }
    v = warp_sum(v);
    if (lane == 0) strand[w] = v;
  }
  __syncthreads();
  const double t = ((strand[0] + strand[1]) + (strand[2] + strand[3])) + ((strand[4] + strand[5]) + (strand[6] + strand[7]));
  __syncthreads();
  return t;
}

// Sum v over the block and store it in part[blockIdx.x].
__device__ __forceinline__ void block_sum_to(double v, double* part) {
  __shared__ double sh[kBlock];
  if (blockDim.x > kBlock) {
    __shared__ double sw[32];
    v = warp_sum(v);
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if (lane == 0) sw[w] = v;
    __syncthreads();
    if (w == 0) {
      const int nw = (blockDim.x + 31) >> 5;
      double t = lane < nw ? sw[lane] : 0.0;
      t = warp_sum(t);
      if (lane == 0) part[blockIdx.x] = t;
    }
    __syncthreads();
    return;
  }
  sh[threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    const double t = warp0_column_sum(sh);
    if (threadIdx.x == 0) part[blockIdx.x] = t;
  }
  __syncthreads();
}

// min and max of values on the integer pipe (dkey order; NaN left out, as fmin / fmax do; atomics
// on the keys, so the result does not depend on the order of the blocks), written straight to
// the pinned host mirror h[60], h[61] by the last block, which leaves the keys empty for the
// next launch.  No further launch and no copy, where two passes with FP64 compares and a copy of the
// scalars took 8 us each and a copy's latency.  key: max, min, blocks done.
struct Range {
  long long mx = LLONG_MIN, mn = LLONG_MAX;

  __device__ __forceinline__ void add(double v) {
    if ((__double_as_longlong(v) & 0x7fffffffffffffffll) > 0x7ff0000000000000ll) return;
    const long long k = dkey(v);
    mx = k > mx ? k : mx;
    mn = k < mn ? k : mn;
  }
  // every thread of a block of whole warps; thread 0 of the last block returns true
  __device__ __forceinline__ bool finish(long long* key, double* h) {
    __shared__ long long smx[32], smn[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const long long a = __shfl_xor_sync(0xffffffffu, mx, o), b = __shfl_xor_sync(0xffffffffu, mn, o);
      mx = a > mx ? a : mx;
      mn = b < mn ? b : mn;
    }
    if ((threadIdx.x & 31) == 0) {
      smx[threadIdx.x >> 5] = mx;
      smn[threadIdx.x >> 5] = mn;
    }
    __syncthreads();
    if (threadIdx.x != 0) return false;
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      mx = smx[w] > mx ? smx[w] : mx;
      mn = smn[w] < mn ? smn[w] : mn;
    }
    atomicMax(key, mx);
    atomicMin(key + 1, mn);
    __threadfence();
    if (atomicAdd(reinterpret_cast<unsigned long long*>(key + 2), 1ull) != gridDim.x - 1) return false;
    __threadfence();
    mx = (long long)atomicExch(reinterpret_cast<unsigned long long*>(key), (unsigned long long)LLONG_MIN);
    mn = (long long)atomicExch(reinterpret_cast<unsigned long long*>(key + 1), (unsigned long long)LLONG_MAX);
    key[2] = 0;
    h[60] = mn == LLONG_MAX ? INFINITY : from_key(mn);    // no number at all: as an empty fmin / fmax
    h[61] = mx == LLONG_MIN ? -INFINITY : from_key(mx);
    return true;
  }
};

// Run f(std::integral_constant<int, K>) with K fixed at compile time for the two
// structured patterns (15 offsets: Kuhn P1, 27: Q1) so that the per-row loops
// unroll completely and all loads of a row are in flight together; 0 = any K.
template <class F>
inline void with_K(int K, F&& f) {
  if (K == 15) f(std::integral_constant<int, 15>{});
  else if (K == 27) f(std::integral_constant<int, 27>{});
  else f(std::integral_constant<int, 0>{});
}

// Programmatic dependent launch between consecutive passes: a pass lets the next one
// launch as soon as all of its blocks run (griddepcontrol.launch_dependents), and the
// next pass issues the loads of data no earlier pass writes before it waits for its
// predecessor's results (griddepcontrol.wait), so those loads overlap the predecessor's
// last wave.  Launched without the attribute, both are no-ops.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Launch kernel k with programmatic dependent launch on `pdl`.
template <class... KArgs, class... Args>
inline cudaError_t launch_pass(bool pdl, void (*k)(KArgs...), dim3 g, dim3 b, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = g;
  cfg.blockDim = b;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k, args...);
}

// out[0] = sum of part[0..n) in a fixed order (one block).
void finalize_sum(afc_problem_s* p, const double* part, int n, double* out);

}  // namespace afc
